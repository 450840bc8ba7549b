"""The Dual EnKF at the largest grids with so many members that each grid has
one CTA: up to 1024 nodes, a thread each and none to spare for a halo."""
import numpy as np
import pytest

import oracle as O
from helpers import rel_err

pytestmark = pytest.mark.gpu

L, NU, DT = 12.8, 1 / 200, 2e-4


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2012_10091_gb300 import mgenkf
    return mgenkf


def _pair(M, nf, ne):
    rng = np.random.default_rng(nf + ne)
    theta0 = np.stack([rng.normal(0.0, 0.05, ne), rng.normal(0.3, 0.05, ne)], axis=1)
    x = np.arange(nf) / nf
    fine0 = 1.0 + 0.2 * np.sin(2 * np.pi * x)
    mem0 = 1.0 + 0.1 * rng.standard_normal((ne, 1)) + 0.2 * np.sin(2 * np.pi * x + 0.3)
    obs = np.arange(1, 13)
    mg = O.DualMGEnKF(nf, 1, L, DT, NU, fine0, mem0, theta0, [0.1, 0.3], obs, 0.05, 7, 1e-6)
    g = M.DualMGEnKF(nf, 1, ne, obs, L, DT, NU, 0.05, 1e-6, 7)
    g.set_state(fine0, mem0, theta0, [0.1, 0.3], 0.0)
    return g, mg, rng


@pytest.mark.parametrize("nf,ne", [(1018, 77), (1019, 77), (1023, 80), (1024, 80), (1024, 256)])
def test_free_run_matches_oracle(M, nf, ne):
    g, mg, _ = _pair(M, nf, ne)
    mg.free_run(33)
    g.free_run(33)
    fine, mem, _, _ = g.get_state()
    g.close()
    # 33 steps x 3 stages of a few roundings of values near 1, each 1.1e-16
    assert np.max(np.abs(fine - mg.fine)) <= 1e-12
    assert np.max(np.abs(mem - mg.members)) <= 1e-12


def test_cycle_matches_oracle(M):
    g, mg, rng = _pair(M, 1024, 80)
    for _ in range(2):
        yo = 1.0 + 0.2 * np.sin(2 * np.pi * np.arange(1, 13) / 1024) + 0.05 * rng.standard_normal(12)
        mg.cycle_step(10, yo)
        g.cycle(10, yo)
    fine, mem, th, tf = g.get_state()
    g.close()
    # as the parameter update's tests: condition below 1e5, FP64 on both sides
    for got, ref in ((th, mg.theta), (tf, mg.theta_fine), (mem, mg.members), (fine, mg.fine)):
        assert rel_err(got, ref) < 1e-10
