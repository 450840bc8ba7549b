"""The FP64 member update for every number of columns per warp, at points and
members that leave a remainder of its tiles."""
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


# coarse points, members: 1 column per warp (129: one point in the second CTA),
# then 2 .. 8 columns on 152 SMs, ne + 1 not a multiple of most of them
@pytest.mark.parametrize("nc,ne", [(40, 2), (129, 9), (200, 100), (3800, 40), (1024, 64), (2600, 31), (3000, 30),
                                   (3000, 128), (2048, 63)])
def test_update_matches_oracle(M, nc, ne):
    w = W.burgers_custom(nc, 1, ne, 12, cycles=1, obs_kind="random")
    inp = W.make_inputs(w)
    yo = W.sample_truth(w, inp["truth0"], inp["obs_idx"], inp["obs_var"]) + W.observation_noise(w, 0)
    g = M.MGEnKF.from_workload(w)
    g.set_state(inp["fine0"], inp["members0"])
    g.analyse(yo)
    g.prolong_correct()
    assert g.sync() == 0
    fine, mem = g.get_state()
    g.close()
    mg = O.MGEnKF(w.model, w.nf, w.ratio, w.length, w.dt, inp["fine0"], inp["members0"], inp["obs_idx"],
                  inp["obs_var"], w.sigma, w.seed, nu=w.nu)
    assert mg.analyse(yo) == 0
    mg.prolong_correct()
    # sums of at most 128 products and a solve of that order: 1e-12 of the state, hundredfold
    for got, ref in ((fine, mg.fine), (mem, mg.members)):
        assert np.max(np.abs(got - ref.reshape(got.shape))) <= 1e-10 * np.max(np.abs(ref))
