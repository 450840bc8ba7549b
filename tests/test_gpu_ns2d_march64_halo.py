"""The FP64 NS-2D row march with halo columns in long runs of rows: strips
narrower than the CTA, of many grids (few grids get runs too short for a thread
past its strip's columns to fill in a halo node)."""
import numpy as np
import pytest

import oracle as O
from paper_2012_10091_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STEPS = 2


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2012_10091_gb300 import mgenkf
    return mgenkf


def _inputs(nc, ratio, ne):
    w = W.ns2d_shear(nf=nc * ratio, ratio=ratio, ne=ne, n_probes=4, precision="fp64",
                     delta=0.02 * max(1.0, 128.0 / nc))
    return w, W.make_inputs(w)


def _check(got, x0, w, n):
    ref = O.ns2d_rk3(x0.reshape(-1, 4, n, n), w.length / n, w.gamma, w.nu, w.prandtl, w.dt, STEPS)
    # some roundings of 2^-53 of the largest plane (E, about 20) per step: 1e-12
    # of it leaves two orders of magnitude
    assert np.max(np.abs(got.reshape(ref.shape) - ref)) <= 1e-12 * np.max(np.abs(ref))


# members' strips and rows per run, fine run: 2 x 68 columns, 34 rows, 3 x 91; 2 x
# 72, 24 and 3 x 96; 2 x 96, 39 and 6 x 128; 1 x 72, 36 and 2 x 72
@pytest.mark.parametrize("nc,ratio,ne", [(136, 2, 48), (144, 2, 32), (192, 4, 32), (72, 2, 200)])
def test_handle_forecast_matches_oracle(M, nc, ratio, ne):
    w, inp = _inputs(nc, ratio, ne)
    g = M.MGEnKF.from_workload(w, precision="fp64")
    g.set_state(inp["fine0"], inp["members0"])
    g.forecast(STEPS)
    assert g.sync() == 0
    fine, mem = g.get_state()
    g.close()
    _check(fine, inp["fine0"], w, w.nf)
    _check(mem, inp["members0"], w, w.nc)


# 3 x 96 columns, 32 rows; 4 x 98, 36; 3 x 88, 44
@pytest.mark.parametrize("n,grids", [(288, 16), (392, 10), (264, 50)])
def test_stateless_forecast_matches_oracle(M, n, grids):
    import torch
    w, inp = _inputs(n, 1, grids)
    x = torch.tensor(inp["members0"], dtype=torch.float64, device="cuda")
    M.mgk_forecast(M.MGENKF_NS2D, M.MGENKF_FP64, x, grids, n, w.length, w.dt, w.nu, w.gamma, w.prandtl, nsteps=STEPS)
    torch.cuda.synchronize()
    _check(x.cpu().numpy(), inp["members0"], w, n)
