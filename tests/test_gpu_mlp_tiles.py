"""The residual network's one-pass kernel at the edges of its tiles: batches below,
at and above a 32-row tile and above one tile per block, inputs narrower and
wider than the 128 staged columns, against the FP64 oracle with BF16 weights.

Bars: those of the oracle test at one size (forward 1e-4, gradients 2e-4 of the
largest entry); FP32 sums of up to 300 products and of the batch stay below them.
"""
import numpy as np
import pytest

from oracle import learned as ol

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("d_in,batch", [(7, 1), (54, 31), (54, 33), (128, 32), (130, 65), (300, 40), (54, 6001)])
def test_forward_and_gradients_over_tiles(d_in, batch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_01863_gb300 import bse
    ctx = bse.Context(0, torch.cuda.current_stream().cuda_stream)
    p0 = bse.mlp_flatten(ol.init_params(d_in, seed=5))
    mlp = ctx.bse_mlp_create(d_in, batch, p0)
    rng = np.random.default_rng(d_in + batch)
    X = rng.standard_normal((batch, d_in)).astype(np.float32)
    Y = rng.standard_normal((batch, 2)).astype(np.float32)
    Xd, Yd = torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda()
    out = torch.full((batch, 2), float("nan"), device="cuda")
    ctx.bse_mlp_forward(mlp, batch, Xd.data_ptr(), out.data_ptr())
    g, loss = ctx.bse_mlp_gradients(mlp, batch, Xd.data_ptr(), Yd.data_ptr())
    g2, loss2 = ctx.bse_mlp_gradients(mlp, batch, Xd.data_ptr(), Yd.data_ptr())
    assert np.array_equal(g, g2) and loss == loss2
    params = bse.mlp_unflatten(p0, d_in)
    for layer in params:
        layer[0] = torch.from_numpy(layer[0]).to(torch.bfloat16).to(torch.float64).numpy()
    ref, cache = ol.forward(params, X.astype(np.float64))
    rl, dout = ol.loss_and_grad_out(ref, Y.astype(np.float64))
    rg = bse.mlp_flatten(ol.backward(params, cache, dout))
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-4 * np.abs(ref).max()
    assert loss == pytest.approx(rl, rel=1e-4)
    assert np.abs(g - rg).max() <= 2e-4 * np.abs(rg).max()
    mlp.free()
    ctx.close()
