"""Tensor-core backward pass of the learned correction where its tiling can go
wrong: two 128-pixel strips with a ragged second one, four-row and two-row
forward tiles, several runs of rows per strip, and arrays that do not start on
a 16-byte boundary."""
import numpy as np
import pytest

import oracle as O
from test_gpu_cnn import _bf16, _case, _gpu, _rel

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


def _dev(a, offset=0):
    """A float32 copy on the device, starting `offset` values into its allocation."""
    import torch
    flat = torch.empty(a.size + offset, dtype=torch.float32, device="cuda")
    view = flat[offset:].view(a.shape)
    view.copy_(torch.tensor(a, dtype=torch.float32))
    return view


def _round(a):
    import torch
    return torch.tensor(np.asarray(a, np.float64)).to(torch.bfloat16).to(torch.float64).numpy()


def _reference(pq, dC, xs, target, stats):
    """Loss and gradients of one sample in FP64, from activations rounded to
    BF16 where the GPU rounds them."""
    s_out = np.asarray(stats["s_out"], np.float32).astype(np.float64)[:, None, None]
    mu, sc = (np.asarray(stats[k], np.float32).astype(np.float64)[:, None, None] for k in ("mu_in", "s_in"))
    f32 = [np.asarray(a, np.float32).astype(np.float64) for a in (dC, xs, target)]
    nc = dC.shape[-1]
    a0 = _round((np.concatenate(f32[:2]) - mu) / sc)
    a1 = _round(np.maximum(O.conv3x3(a0, pq["W1"], pq["b1"]), 0.0))
    a2 = _round(np.maximum(O.conv3x3(a1, pq["W2"], pq["b2"]), 0.0))
    base = O.prolong_add(f32[0].reshape(-1), np.zeros(4 * (4 * nc) ** 2), 2, 4, nc, 4).reshape(target.shape)
    r = (base + O.pixel_shuffle4(O.conv3x3(a2, pq["W3"], pq["b3"])) * s_out - f32[2]) / s_out
    da2, dW3, db3 = O.conv3x3_bwd(a2, pq["W3"], O.pixel_unshuffle4(2.0 * r / r.size))
    da1, dW2, db2 = O.conv3x3_bwd(a1, pq["W2"], da2 * (a2 > 0))
    _, dW1, db1 = O.conv3x3_bwd(a0, pq["W1"], da1 * (a1 > 0), want_din=False)
    return float((r * r).mean()), dict(W1=dW1, b1=db1, W2=dW2, b2=db2, W3=dW3, b3=db3)


# (4, 1), (5, 2): maps narrower than a tile by far; (129, 1): a strip of one
# pixel; (130, 5): four-row tiles, ten strips; (64, 3): one strip
@pytest.mark.parametrize("nc,B", [(4, 1), (5, 2), (64, 3), (129, 1), (130, 5)])
def test_gradients_over_strips_and_rows(M, nc, B):
    """Against FP64 gradients of the same BF16 activations and weights.  What
    remains is FP32 accumulation and the activations whose FP32 sum lands on
    the other side of a BF16 rounding boundary: sums of up to 288 products err
    by about 2^-24 sqrt(288) < 2^-19 of their size, so about 2^-19 / 2^-8 = 1
    in 2048 activations moves by one BF16 ulp (2^-8), a norm-wise change of
    2^-8 / sqrt(2048) < 1e-4 per layer: 1e-3 over the three layers, and for the
    weight gradients that cancel, whose entries are a tenth of their terms."""
    params, stats, dC, xs, target = _case(nc, B, 40 + nc)
    cnn = _gpu(M, nc, B, params, stats)
    loss = _dev(np.zeros(1))
    cnn.loss_grad(_dev(dC), _dev(xs), _dev(target), B, loss)
    g = M.unflatten_cnn(cnn.get_params()[1])
    cnn.close()
    pq = {k: (_bf16(v) if k.startswith("W") else np.asarray(v, np.float32).astype(np.float64))
          for k, v in params.items()}
    refs = [_reference(pq, dC[b], xs[b], target[b], stats) for b in range(B)]
    tot_loss = sum(r[0] for r in refs) / B
    assert abs(float(loss.item()) - tot_loss) <= 1e-4 * tot_loss
    for k in params:
        ref = sum(r[1][k] for r in refs) / B
        assert _rel(g[k], ref) < 1e-3, (k, _rel(g[k], ref))


@pytest.mark.parametrize("nc,B", [(20, 2), (130, 1)])
def test_unaligned_arrays_give_the_same_bits(M, nc, B):
    params, stats, dC, xs, target = _case(nc, B, 60 + nc)
    cnn = _gpu(M, nc, B, params, stats)
    out = []
    for off in (0, 1):
        base = np.full((B, 4, 4 * nc, 4 * nc), 0.5)
        res, acc, loss = _dev(base, off), _dev(base, off), _dev(np.zeros(1))
        d, x, t = _dev(dC, off), _dev(xs, off), _dev(target, off)
        cnn.forward(d, x, B, res)
        cnn.forward(d, x, B, acc, accumulate=True)
        cnn.loss_grad(d, x, t, B, loss)
        out.append([res.cpu().numpy(), acc.cpu().numpy(), float(loss.item()), cnn.get_params()[1]])
    cnn.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
    np.testing.assert_allclose(out[0][1], out[0][0] + np.float32(0.5), rtol=0, atol=1e-6 * (1 + np.abs(out[0][0]).max()))
