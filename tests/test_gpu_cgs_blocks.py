"""Reorthogonalised recursions where the Gram-Schmidt kernels split their work.

Sizes: vectors shorter than one 32-entry block of the update, one block of the
products per vector, several of them with a ragged last one, and several chains.
The oracle runs the same recursion on the host with the library's H.

Bars: FP64, relative 1e-10 in a and b, the bar of the other recursion tests.
"""
import numpy as np
import pytest

from oracle import haydock as oh
from oracle import interp as oi
from paper_1602_01863_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nv,nc,n,nd,chains,steps", [
    (1, 1, 3, 1, 1, 8),     # N = 27
    (2, 2, 3, 2, 3, 25),    # N = 864: one block per vector, three chains
    (1, 3, 5, 3, 1, 20),    # N = 10125: ten blocks per vector, 13 entries in the last 32
    (3, 3, 7, 3, 2, 20),    # N = 83349: as many blocks as the SMs take
])
def test_cgs2_matches_host_recursion(nv, nc, n, nd, chains, steps):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_01863_gb300 import bse
    torch.cuda.set_device(0)
    ctx = bse.Context(0, torch.cuda.current_stream().cuda_stream)
    m = synth.draw_model(73, nv, nc)
    co = ctx.bse_build_coarse(m, n, bse.PREC_F64)
    it = ctx.bse_interp_setup(co, nd, bse.SCHEME_M3, 0.8, bse.PREC_F64)
    I = oi.Interp(m, n, nd, width=0.8, build_dense_kc=False)

    def apply(v):
        x = torch.from_numpy(np.ascontiguousarray(v.reshape(1, -1))).cuda()
        y = torch.empty_like(x)
        ctx.bse_apply_h(it, 1, x.data_ptr(), y.data_ptr())
        return y.cpu().numpy().reshape(v.shape)

    dirs = np.eye(3)[:chains]
    a, b, pn2, st, rc = ctx.bse_haydock_run([it], [chains], dirs, steps, bse.REORTH_CGS2)
    assert rc == 0
    for ch in range(chains):
        ra, rb, rp, _ = oh.haydock(apply, I.dipole(dirs[ch]), steps, "cgs2")
        assert np.max(np.abs(a[ch] - ra) / np.abs(ra)) < 1e-10
        assert np.max(np.abs(b[ch, 1:] - rb[1:]) / np.abs(rb[1:])) < 1e-10
    it.free()
    co.free()
    ctx.close()
