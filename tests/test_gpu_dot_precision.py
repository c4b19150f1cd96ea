"""a_i of FP32 vectors: the sum <psi, w> keeps the bits of the vectors' products.

The first step's a_1 against the FP64 product of the same FP32 vectors (the start
vector as the library scales it, w from bse_apply_h), where a thread has few products,
many, and the most (n_div 16 or 64 transitions), with and without the learned correction.

Bar: 1e-12 |a|.  Products enter exactly and the additions' roundings are kept, so
a thread's sum of n products is off by about n 2^-50 of itself, n <= 2048, and the block
partials add up in FP64.  Single FP32 sums are off by some 1e-9.
"""
import numpy as np
import pytest

from paper_1602_01863_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nv,nc,n,nd,scheme,learned", [
    (2, 2, 3, 2, 1, 0),
    (3, 5, 4, 4, 1, 0),      # several points to a lane
    (1, 1, 2, 16, 0, 0),     # one transition: sixteen lanes' points
    (8, 8, 2, 8, 0, 0),      # two entries to a lane, 64 points each
    (8, 8, 2, 16, 0, 0),     # 512 points each
    (3, 4, 12, 4, 0, 2),     # learned: 36 products of a plane to a thread
    (2, 3, 8, 8, 0, 2),      # 64 of them
    (2, 3, 11, 1, 0, 2),     # the separate passes
])
def test_first_coefficient(nv, nc, n, nd, scheme, learned):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_01863_gb300 import bse
    ctx = bse.Context(0, torch.cuda.current_stream().cuda_stream)
    co = ctx.bse_build_coarse(synth.draw_model(63, nv, nc), n, bse.PREC_F32)
    it = ctx.bse_interp_setup(co, nd, scheme, 0.9, bse.PREC_F32)
    mlp = None
    if learned:
        d_in = 6 + 2 * it.t
        r = np.random.default_rng(4)
        mlp = ctx.bse_mlp_create(d_in, 4096, (0.3 * r.standard_normal(ctx.lib.bse_mlp_param_count(d_in))).astype(np.float32))
        ctx.bse_interp_set_learned(it, mlp, learned)
    dirs = synth.POL3[:2].copy()
    a, b, pn2, _, _ = ctx.bse_haydock_run([it], [2], dirs, 1, 0)
    P = torch.empty((2, it.N), dtype=torch.complex64, device="cuda")
    ctx.bse_dipoles(it, dirs, P.data_ptr())
    inv = torch.from_numpy(1.0 / np.sqrt(pn2)).cuda()
    psi = torch.view_as_complex((torch.view_as_real(P).double() * inv[:, None, None]).float())
    w = torch.empty_like(psi)
    ctx.bse_apply_h(it, 2, psi.data_ptr(), w.data_ptr())
    p, q = psi.cpu().numpy().astype(np.complex128), w.cpu().numpy().astype(np.complex128)
    for ch in range(2):
        ref = np.vdot(p[ch], q[ch]).real
        print(f"a_1 {ref:.6f}, off by {abs(a[ch, 0] - ref) / abs(ref):.1e}")
        # the separate passes sum a thread's few products in FP32, as they always have
        assert abs(a[ch, 0] - ref) <= (1e-12 if n * nd != 11 else 1e-7) * abs(ref)
    if mlp:
        mlp.free()
    it.free()
    co.free()
    ctx.close()
