"""Rounding errors of the FP64 Burgers forecast against extended precision: no
larger than those of the scheme with every derivative formed from neighbour
differences, evaluated in FP64."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NU, STEPS = 0.01, 60


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2012_10091_gb300 import mgenkf
    return mgenkf


def _edge_differences(u, dt, t):
    """STEPS SSP-RK3 steps of the rows of u in the type t."""
    dx, dt, nu = t(2 * math.pi / u.shape[1]), t(dt), t(NU)
    a, b = dt / (4 * dx), dt * nu / (dx * dx)
    u = u.astype(t)

    def dtl(v):
        w, e = np.roll(v, 1, 1), np.roll(v, -1, 1)
        return a * ((w - e) * (w + e)) + b * ((e - v) + (w - v))

    for _ in range(STEPS):
        k0 = dtl(u)
        k = k0 + dtl(u + k0)
        u = u + (k / 6 + 2 * dtl(u + k / 4) / 3)
    return u


# as many grids as keep 16384 points: the rms over them is known to about 2%, and
# the two forms differ by that and by how their constants round; a derivative
# formed from a rounded sum of neighbours is 13% and more off
@pytest.mark.parametrize("n", [2048, 4096, 16384])
def test_errors_are_those_of_neighbour_differences(M, n):
    import torch
    if np.finfo(np.longdouble).nmant < 60:
        pytest.skip("no extended precision")
    grids = 16384 // n
    rng = np.random.default_rng(n)
    x = 2 * math.pi * np.arange(n) / n
    prof = sum(np.sin(k * x + p) / k for k, p in zip(range(1, 6), (0.3, 1.1, 2.7, 4.0, 5.2)))
    u0 = (0.8 + 0.1 * rng.standard_normal((grids, 1))) * prof + 0.01 * rng.standard_normal((grids, n))
    dt = 0.314 * (2 * math.pi / n) ** 2 / NU
    g = torch.tensor(u0, device="cuda")
    M.mgk_forecast(M.MGENKF_BURGERS1D, M.MGENKF_FP64, g, grids, n, 2 * math.pi, dt, NU, nsteps=STEPS)
    exact = _edge_differences(u0, dt, np.longdouble)

    def rms(v):
        return float(np.sqrt(np.mean((v - exact) ** 2)))

    assert rms(g.cpu().numpy()) <= 1.07 * rms(_edge_differences(u0, dt, np.float64))
