"""The blocked FP64 gain solve at the edges of its blocks and clusters, through
the allocation-free entry point (n = members) and through a direct-form handle
(n = observations): one block, a ragged last block, more blocks in a column than
workers, the change of cluster size and the largest order."""
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


@pytest.mark.parametrize("n", [2, 15, 16, 17, 31, 33, 100, 112, 113, 128])
def test_ensemble_form_orders(M, n):
    import torch
    ny, sigma = 40, 0.3
    rng = np.random.default_rng(n)
    Y, Z = rng.standard_normal((n, ny)) / np.sqrt(n), rng.standard_normal((n + 1, ny))
    T = torch.zeros((n + 1, n), dtype=torch.float64, device="cuda")
    info = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    M.mgk_gain_ensemble_noalloc(torch.tensor(Y, device="cuda"), torch.tensor(Z, device="cuda"), n, ny, sigma, T, info)
    assert int(info.item()) == 0
    S = np.eye(n) + Y @ Y.T / sigma ** 2
    ref = np.linalg.solve(S, Y @ Z.T / sigma ** 2).T
    # backward-stable solve: n 2^-53 cond(S) relative, cond(S) < 1e3 here
    assert np.linalg.norm(T.cpu().numpy() - ref) <= 1e-11 * np.linalg.norm(ref)


@pytest.mark.parametrize("ny", [1, 16, 130, 240, 241, 256, 257])
def test_direct_form_orders(M, ny):
    w = W.burgers_custom(1024, 4, 24, ny, cycles=1, obs_kind="random")
    inp = W.make_inputs(w)
    yo = W.sample_truth(w, inp["truth0"], inp["obs_idx"], inp["obs_var"]) + W.observation_noise(w, 0)
    g = M.MGEnKF.from_workload(w, gain_form=M.MGENKF_GAIN_DIRECT)
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
    for got, ref in ((fine, mg.fine), (mem, mg.members)):
        assert np.max(np.abs(got - ref.reshape(got.shape))) <= 1e-10 * np.max(np.abs(ref))


def test_indefinite_matrix_is_reported_from_any_block(M):
    """An observation variance of zero with more observations than Ne - 1 makes
    the direct form's matrix singular: its rounded pivots past the rank are not
    all positive.  The state stays as it was."""
    w = W.burgers_custom(512, 4, 6, 120, cycles=1, obs_kind="random", sigma=0.0)
    inp = W.make_inputs(w)
    yo = W.sample_truth(w, inp["truth0"], inp["obs_idx"], inp["obs_var"])
    g = M.MGEnKF.from_workload(w, gain_form=M.MGENKF_GAIN_DIRECT)
    g.set_state(inp["fine0"], inp["members0"])
    g.analyse(yo)
    g.prolong_correct()
    assert g.sync() == 4
    fine, mem = g.get_state()
    g.close()
    np.testing.assert_array_equal(fine, inp["fine0"])
    np.testing.assert_array_equal(mem, inp["members0"])
