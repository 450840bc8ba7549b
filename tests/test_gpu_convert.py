"""State conversions between FP64 and FP32 (a mixed-precision handle's set_state
and get_state) bit for bit: ties, subnormals, zeros of both signs, the edges of
the FP32 range, infinities and NaN, and a length that leaves a remainder."""
import numpy as np
import pytest

from paper_2012_10091_gb300 import workloads as W

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


@pytest.mark.parametrize("nf,ne", [(1028, 3), (16384, 40)])
def test_conversions_are_the_formats_own(M, nf, ne):
    w = W.burgers_custom(nf, 4, ne, 8, cycles=1, precision="mixed")
    rng = np.random.default_rng(nf)
    tiny, big = np.finfo(np.float32).tiny, np.finfo(np.float32).max
    special = np.array([0.0, -0.0, tiny, -tiny, tiny * (1 - 2.0 ** -24), tiny * 0.3, 2.0 ** -149, 2.0 ** -150, 1e-300, big, -big,
                        np.nextafter(float(big) * (1 + 2.0 ** -25), 0.0), float(big) * (1 + 2.0 ** -24), 1e39, np.inf,
                        -np.inf, np.nan, 1.0 + 2.0 ** -24, 1.0 + 3 * 2.0 ** -24, -1.0 - 2.0 ** -24 - 2.0 ** -50])

    def values(n):
        x = rng.standard_normal(n) * 10.0 ** rng.uniform(-46, 40, n)
        x[: n // 4] = (rng.integers(0, 2 ** 24, n // 4) + 0.5) * 2.0 ** rng.integers(-160, 110, n // 4)  # ties
        x[n - special.size:] = special
        return x

    fine, mem = values(nf), values(ne * (nf // 4)).reshape(ne, nf // 4)
    g = M.MGEnKF.from_workload(w, precision="mixed")
    g.set_state(fine, mem)
    got_f, got_m = g.get_state()
    g.close()
    with np.errstate(all="ignore"):
        ref_f, ref_m = fine.astype(np.float32).astype(np.float64), mem.astype(np.float32).astype(np.float64)
    for got, ref in ((got_f, ref_f), (got_m, ref_m)):
        got = np.asarray(got).reshape(ref.shape)
        same = (got.view(np.uint64) == ref.view(np.uint64)) | (np.isnan(got) & np.isnan(ref))
        assert same.all(), (got[~same][:4], ref[~same][:4])
