"""The parameter update of the Dual EnKF (a cluster of CTAs that pass their
sums to the first) at the edges of its split of the members: fewer members than
warps, than CTAs times warps, one more, the largest ensemble; several cycles in
a row, each reading the mean that the one before has written."""
import numpy as np
import pytest

import oracle as O
from helpers import rel_err

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


@pytest.mark.parametrize("ne", [2, 7, 8, 63, 64, 65, 129, 256])
def test_parameters_match_oracle(M, ne):
    nf, r, L, nu, dt, sigma, q = 64, 2, 0.8, 1 / 200, 2e-4, 0.05, 1e-5
    rng = np.random.default_rng(ne)
    theta0 = np.stack([rng.normal(0.0, 0.05, ne), rng.normal(0.3, 0.05, ne)], axis=1)
    fine0 = 1.0 + 0.1 * np.sin(2 * np.pi * np.arange(nf) / nf)
    mem0 = 1.0 + 0.05 * rng.standard_normal((ne, 1)) + 0.1 * np.sin(2 * np.pi * np.arange(0, nf, r) / nf)
    obs = np.arange(1, 13)
    mg = O.DualMGEnKF(nf, r, L, dt, nu, fine0, mem0, theta0, [0.05, 0.3], obs, sigma, 7, q)
    g = M.DualMGEnKF(nf, r, ne, obs, L, dt, nu, sigma, q, 7)
    g.set_state(fine0, mem0, theta0, [0.05, 0.3], 0.0)
    for _ in range(4):
        yo = 1.0 + 0.1 * np.sin(2 * np.pi * obs / nf + 0.2) + sigma * rng.standard_normal(obs.size)
        mg.cycle_step(10, yo)
        g.cycle(10, yo)
    fine, mem, th, tf = g.get_state()
    g.close()
    # FP64 on both sides: sums of up to 256 terms and a solve of condition below
    # 1e5 (sigma 0.05, spreads of 0.05), 4 cycles
    for got, ref in ((th, mg.theta), (tf, mg.theta_fine), (mem, mg.members), (fine, mg.fine)):
        assert rel_err(got, ref) < 1e-10
