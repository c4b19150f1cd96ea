"""FP32 buffers of the caller that start on 4 bytes and not on 8 or 16: the pair data,
the network's inputs and outputs.  They hold exactly what aligned ones hold.
"""
import numpy as np
import pytest

from paper_1602_01863_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _at(rows, cols, shift):
    """A [rows, cols] view that starts `shift` floats into its storage."""
    return torch.full((rows * cols + shift,), float("nan"), device="cuda")[shift:].view(rows, cols)


@pytest.mark.parametrize("prec", [0, 1])
def test_unaligned_buffers(prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_01863_gb300 import bse
    ctx = bse.Context(0, torch.cuda.current_stream().cuda_stream)
    co = ctx.bse_build_coarse(synth.draw_model(53, 2, 3), 3, prec)
    it = ctx.bse_interp_setup(co, 2, bse.SCHEME_M1, 1.0, prec)
    t, blocks = it.t, 5
    rng = np.random.default_rng(6)
    kd, kd2 = rng.integers(0, it.Nk, blocks), rng.integers(0, it.Nk, blocks)
    rows, d_in = blocks * t * t, 6 + 2 * t
    mlp = ctx.bse_mlp_create(d_in, rows, (0.1 * rng.standard_normal(ctx.lib.bse_mlp_param_count(d_in))).astype(np.float32))
    out = []
    for shift in (0, 1, 3):
        X, Y, pred = _at(rows, d_in, shift), _at(rows, 2, shift), _at(rows, 2, shift)
        assert X.data_ptr() % 16 == 4 * shift and Y.data_ptr() % 16 == 4 * shift
        ctx.bse_pairs_generate(it, kd, kd2, X.data_ptr(), Y.data_ptr())
        ctx.bse_mlp_forward(mlp, rows, X.data_ptr(), pred.data_ptr())
        g, loss = ctx.bse_mlp_gradients(mlp, rows, X.data_ptr(), Y.data_ptr())
        out.append((X.cpu().numpy(), Y.cpu().numpy(), pred.cpu().numpy(), g, np.array(loss)))
    assert all(np.all(np.isfinite(v)) for v in out[0])
    for o in out[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(out[0], o))
    mlp.free()
    it.free()
    co.free()
    ctx.close()
