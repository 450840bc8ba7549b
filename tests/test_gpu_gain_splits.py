"""The gain products over their K splits: one split, a cluster of 2 to 8, several
splits per CTA, more than a cluster takes, and members that leave a remainder of
the tiles, in FP64 and in double-FP32 (mixed precision)."""
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


# members, observations: splits 1 (a K chunk that is not whole), 2, 4, 8, 16 (two
# per CTA), 32 (four per CTA), 64 (partial sums in memory); 33 members: a tile of
# one row
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("ne,ny", [(7, 45), (33, 300), (20, 515), (16, 1024), (20, 2050), (20, 4096), (7, 8192)])
def test_analysis_matches_oracle(M, precision, ne, ny):
    w = W.burgers_custom(16384 if ny > 2050 else 4096, 16, ne, ny, cycles=1, obs_kind="random")
    inp = W.make_inputs(w)
    yo = W.sample_truth(w, inp["truth0"], inp["obs_idx"], inp["obs_var"]) + W.observation_noise(w, 0)
    g = M.MGEnKF.from_workload(w, precision=precision)
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
    # FP64: a solve and products of that order, 1e-12 of the state, hundredfold.
    # Mixed: BF16 anomalies and T (2^-9 each) on increments below the state
    bound = 1e-10 if precision == "fp64" else 1e-2
    for got, ref in ((fine, mg.fine), (mem, mg.members)):
        assert np.max(np.abs(got - ref.reshape(got.shape))) <= bound * np.max(np.abs(ref))
