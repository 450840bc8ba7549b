"""The FP64 reciprocal of the gain solve's pivots and of the NS-2D densities.
Gain solves of diagonal systems with unit right-hand sides return the pivots'
reciprocals as they are; an NS-2D forecast takes that of every density."""
import numpy as np
import pytest

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


# exponents of the pivots, 1 + y^2: ordinary ones, large ones, both sides of the
# range's end at 2^993, the largest numbers
@pytest.mark.parametrize("lo,hi", [(0, 1), (0, 60), (60, 990), (985, 1000), (1010, 1023)])
def test_pivot_reciprocals(M, lo, hi):
    import torch
    n, wrong, total = 128, 0, 0
    for seed in range(8):
        rng = np.random.default_rng([seed, lo])
        y = np.sqrt(np.exp2(rng.uniform(lo, hi, n)) * (1 - 1e-3))
        t = 2.0 ** -300  # t^2 vanishes beside 1, t times 2^300 is the unit right-hand side
        Y = np.concatenate([np.diag(y), t * np.eye(n)], axis=1)
        Z = np.concatenate([np.zeros((n, n)), np.eye(n) / t], axis=1)
        Z = np.concatenate([Z, Z[:1]])
        T = torch.zeros((n + 1, n), dtype=torch.float64, device="cuda")
        info = torch.full((1,), -1, dtype=torch.int32, device="cuda")
        M.mgk_gain_ensemble_noalloc(torch.tensor(Y, device="cuda"), torch.tensor(Z, device="cuda"), n, 2 * n, 1.0, T,
                                    info)
        assert int(info.item()) == 0
        got, ref = np.diag(T.cpu().numpy()[:n]), 1.0 / (1.0 + y * y)
        units = np.abs(got - ref) / np.spacing(ref)
        assert np.max(units) <= 1.0
        wrong += int(np.count_nonzero(units))
        total += n
    # 2^-16 of a unit beside the last rounding: 1 in 2^15 quotients lies so close
    # to a tie (chance of more than 2 of 1024: below 1e-5)
    assert total == 1024 and wrong <= 2


def test_infinite_density_spreads_no_further_than_its_flux(M):
    """1 / rho is zero at a point of infinite density, so the first two stages of a
    step change its neighbours by finite amounts; the difference of its own
    stages is not a number, which the third stage hands to the nearest points
    and to no others."""
    import torch
    n, h = 16, 1.0 / 16
    g = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    q = np.stack([1.0 + 0.1 * np.sin(2 * np.pi * g[1] * h), 0.1 * np.cos(2 * np.pi * g[0] * h),
                  0.1 * np.sin(2 * np.pi * g[1] * h), np.full((n, n), 20.0)])
    outs = []
    for bad in (False, True):
        x = q.copy()
        if bad:
            x[0, 8, 8] = np.inf
        d = torch.tensor(x[None], device="cuda")
        M.mgk_forecast(M.MGENKF_NS2D, M.MGENKF_FP64, d, 1, n, 1.0, 1e-4, 1e-3, 1.4, 0.72, nsteps=1)
        outs.append(d.cpu().numpy()[0])
    away = np.maximum(np.abs(g[0] - 8), np.abs(g[1] - 8))
    np.testing.assert_array_equal(outs[0][:, away > 3], outs[1][:, away > 3])
    assert np.isfinite(outs[1][:, away > 1]).all()
