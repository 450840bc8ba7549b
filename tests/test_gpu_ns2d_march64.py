"""The FP64 NS-2D row march where its layout can go wrong: narrow grids packed
side by side into a CTA, one strip per grid, several strips with halo columns
(a ragged last one), runs of rows that do not divide the grid."""
import numpy as np
import pytest

import oracle as O
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


# (coarse side, ratio, members): 8 and 32 packed four to a CTA (with an
# incomplete last CTA), 40 packed two to a CTA, 96 and 128 one strip, 136 two
# strips of 68, 264 three strips of 88, 520 five strips of 104
@pytest.mark.parametrize("nc,ratio,ne", [(8, 1, 5), (32, 1, 7), (40, 2, 3), (8, 16, 33), (136, 1, 2), (66 * 4, 1, 2),
                                         (104, 5, 2)])
def test_march_matches_oracle(M, nc, ratio, ne):
    w = W.ns2d_shear(nf=nc * ratio, ratio=ratio, ne=ne, n_probes=4, precision="fp64",
                     delta=0.02 * max(1.0, 128.0 / nc))
    inp = W.make_inputs(w)
    g = M.MGEnKF.from_workload(w, precision="fp64")
    g.set_state(inp["fine0"], inp["members0"])
    g.forecast(3)
    assert g.sync() == 0
    fine, mem = g.get_state()
    g.close()
    h = [w.length / n for n in (w.nf, w.nc)]
    ref_f = O.ns2d_rk3(inp["fine0"].reshape(4, w.nf, w.nf), h[0], w.gamma, w.nu, w.prandtl, w.dt, 3).reshape(-1)
    ref_m = O.ns2d_rk3(inp["members0"].reshape(ne, 4, nc, nc), h[1], w.gamma, w.nu, w.prandtl, w.dt, 3).reshape(ne, -1)
    # three steps of rounding at 2^-53 of the largest plane (E, about 20): 1e-12
    # of it leaves two orders of magnitude
    for got, ref in ((fine, ref_f), (mem, ref_m)):
        assert np.max(np.abs(got - ref)) <= 1e-12 * np.max(np.abs(ref))
