"""The loss of the learned correction divides by the output scale: scales whose
reciprocal over- or underflows, and differences that are not finite."""
import numpy as np
import pytest

from test_gpu_cnn import _case, _gpu
from test_gpu_cnn_tc import _dev, _reference

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


def _loss(M, nc, params, stats, dC, xs, target):
    import torch
    cnn = _gpu(M, nc, 1, params, stats)
    out = torch.zeros(1, dtype=torch.float32, device="cuda")
    cnn.loss_grad(_dev(dC), _dev(xs), _dev(target), 1, out)
    torch.cuda.synchronize()
    return float(out.item())


# a subnormal scale (its differences are multiples of 1.4e-45, 1.4e-6 of it),
# the largest scales, and ordinary ones
@pytest.mark.parametrize("scale", [1e-39, 1e-33, 1.0, 1e33, 1e38])
def test_loss_for_extreme_scales(M, scale):
    nc = 8
    params, stats, dC, xs, target = _case(nc, 1, 5)
    params["W3"] *= 0.05
    params["b3"] *= 0.05
    stats["s_out"] = np.full(4, scale)
    dC[...] = 0.0
    target *= 0.5 * scale
    loss, _ = _reference(params, dC[0], xs[0], target[0], stats)
    # the loss is a sum over 4096 values of order one in FP32; the forward pass is
    # that of the reference
    assert _loss(M, nc, params, stats, dC, xs, target) == pytest.approx(loss, rel=1e-4)


def test_infinite_difference_gives_infinite_loss(M):
    nc = 8
    params, stats, dC, xs, target = _case(nc, 1, 6)
    target[0, 2, 7, 9] = np.inf
    assert _loss(M, nc, params, stats, dC, xs, target) == np.inf
