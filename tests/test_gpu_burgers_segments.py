"""FP64 Burgers forecasts cut into halo'd segments (members and fine run in
shared launches, grids that are one segment as rings) against the oracle."""
import math

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


# (coarse points, ratio, members, steps): segments on both grids; a single
# segmented launch with its copy back; more, and a prime number of, launches
# than steps divide into; ragged lengths; rings beside a segmented fine run;
# rings alone; halos wider than the grid
@pytest.mark.parametrize("nc,ratio,ne,steps", [(64, 4, 32, 20), (130, 8, 10, 1), (130, 8, 10, 41), (37, 7, 3, 53),
                                               (1000, 8, 100, 25), (8, 16, 300, 20), (9, 3, 2, 31), (2048, 4, 150, 7)])
def test_segmented_forecast_matches_oracle(M, nc, ratio, ne, steps):
    nf = nc * ratio
    dx, nu = 2 * math.pi / nf, 0.01
    w = W.burgers_custom(nf, ratio, ne, 4, dt=min(1e-3, 0.3 * dx * dx / nu, 0.5 * dx))
    inp = W.make_inputs(w)
    g = M.MGEnKF.from_workload(w)
    g.set_state(inp["fine0"], inp["members0"])
    g.forecast(steps)
    assert g.sync() == 0
    fine, mem = g.get_state()
    g.close()
    for got, x0, n in ((fine[None], inp["fine0"][None], nf), (mem, inp["members0"], nc)):
        ref = O.burgers_rk3(x0, w.length / n, w.nu, w.dt, steps)
        # one rounding of 2^-53 per stage and point, amplified at most by the
        # scheme's growth: far below 1e-12 over some tens of steps
        assert np.max(np.abs(got - ref)) <= 1e-12 * np.max(np.abs(ref))
