"""The FP32 NS-2D column march over its layouts: pairs of row segments (an odd
count leaves the last one alone), every pitch of the shared rows, one band and
several with halo columns, ragged bands and segments; it agrees with the tile
kernel bit for bit."""
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


# (coarse side, ratio, members); choices: 32 rows wide, 256 rows (one segment),
# 20 rows and 48 rows in narrow bands.  8 .. 32 points: 32 threads, segments no
# longer than the register windows' first block; 40, 64: 64; 96: 96; 104: 128;
# 136: 192 wide, two narrow bands of 74; 208, 256: 256 wide (the widest single
# band), 264: two wide bands; members 1 and 3: odd numbers of segments
@pytest.mark.parametrize("nc,ratio,ne", [(8, 1, 2), (8, 4, 3), (40, 2, 3), (64, 2, 2), (96, 1, 3), (104, 2, 3), (136, 1, 2),
                                         (256, 1, 2), (264, 1, 3)])
def test_march_agrees_with_the_tile_kernel(M, nc, ratio, ne):
    w = W.ns2d_shear(nf=nc * ratio, ratio=ratio, ne=ne, n_probes=4, precision="mixed",
                     delta=0.02 * max(1.0, 128.0 / nc))
    inp = W.make_inputs(w)
    g = M.MGEnKF.from_workload(w, precision="mixed")
    default = g.forecast_choice()
    for steps in (1, 2):
        ref = None
        for choice in ((-1, -1), (0, 4), (4, 0), (7, 15), (14, 7), default):
            g.set_forecast_choice(*choice)
            g.set_state(inp["fine0"], inp["members0"])
            g.forecast(steps)
            assert g.sync() == 0
            got = g.get_state()
            if ref is None:
                ref = got
            np.testing.assert_array_equal(got[0], ref[0])
            np.testing.assert_array_equal(got[1], ref[1])
    g.close()
