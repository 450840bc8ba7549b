"""The inlet forecast of the Dual EnKF where its layout can go wrong: one CTA
per grid, clusters of 2, 4 and 8 with unequal parts, more grids than SMs, one
step, and step counts around the 32 whose inlet values are formed together."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2012_10091_gb300 import mgenkf
    return mgenkf


# fine nodes, ratio, members: 8 coarse nodes; 122 and 123 nodes: one CTA of 128
# threads, two CTAs; 245 and 489: 4 and 8 CTAs with a shorter last one; 1024:
# the largest; 200 members of 245 nodes: one CTA each
@pytest.mark.parametrize("nf,r,ne,steps", [(16, 2, 3, 33), (122, 1, 2, 64), (123, 1, 5, 1), (245, 1, 4, 65), (245, 1, 200, 2),
                                           (489, 1, 2, 32), (1024, 4, 3, 31), (976, 2, 3, 33)])
def test_free_run_on_clusters_matches_oracle(M, nf, r, ne, steps):
    L, nu, dt = 10.0, 1 / 200, 4e-4
    rng = np.random.default_rng(nf)
    theta0 = np.stack([rng.normal(0.0, 0.05, ne), rng.normal(0.3, 0.05, ne)], axis=1)
    x = np.arange(nf) / nf
    fine0 = 1.0 + 0.2 * np.sin(2 * np.pi * x)
    mem0 = 1.0 + 0.1 * rng.standard_normal((ne, 1)) + 0.2 * np.sin(2 * np.pi * x[::r] + 0.3)
    obs = np.arange(1, 5)
    mg = O.DualMGEnKF(nf, r, L, dt, nu, fine0, mem0, theta0, [0.1, 0.3], obs, 0.05, 7, 1e-6)
    g = M.DualMGEnKF(nf, r, ne, obs, L, dt, nu, 0.05, 1e-6, 7)
    g.set_state(fine0, mem0, theta0, [0.1, 0.3], 0.0)
    for n in (steps, 1):
        mg.free_run(n)
        g.free_run(n)
        fine, mem, _, _ = g.get_state()
        # at most 66 steps x 3 stages of a few roundings of values near 1, each
        # 1.1e-16: below 1e-13
        assert np.max(np.abs(fine - mg.fine)) <= 1e-12
        assert np.max(np.abs(mem - mg.members)) <= 1e-12
