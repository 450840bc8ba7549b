"""Stateless FP64 Burgers forecasts of one to three steps, on each of the routes
between which their plan chooses: rings of one to eight points per thread, whole
grids in place (a CTA or a cluster each), segments with a second buffer."""
import math

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


@pytest.mark.parametrize("n,grids,steps", [(4, 1, 1), (5, 300, 2), (384, 7, 1), (1000, 2000, 1), (1023, 3, 1), (2047, 5, 1),
                                           (2048, 64, 3), (4093, 1, 1), (4093, 300, 1), (4096, 300, 2), (8192, 2, 1),
                                           (12288, 64, 1), (16384, 64, 1), (32768, 1, 3)])
def test_few_steps_match_oracle(M, n, grids, steps):
    import torch
    nu, L = 0.01, 2 * math.pi
    dt = min(1e-3, 0.3 * (L / n) ** 2 / nu)
    x = np.arange(n) / n
    u0 = np.sin(L * x + np.arange(grids)[:, None]) + 0.3
    u = torch.tensor(u0, device="cuda")
    M.mgk_forecast(M.MGENKF_BURGERS1D, M.MGENKF_FP64, u, grids, n, L, dt, nu, nsteps=steps)
    torch.cuda.synchronize()
    ref = O.burgers_rk3(u0, L / n, nu, dt, steps)
    # a few roundings of 2^-53 per stage over at most three steps
    assert np.max(np.abs(u.cpu().numpy() - ref)) <= 1e-13 * np.max(np.abs(ref))
