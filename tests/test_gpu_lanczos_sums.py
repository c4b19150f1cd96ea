"""Lanczos coefficients summed by every block of the update and scale kernels.

The recursion over vector lengths with one block, several, and more partials than
threads, with and without reorthogonalisation, against the same recursion in
64 bits with the library's own H application (FP64: 1e-12 of the largest coefficient, a few
roundings of sums of N products per step over 6 steps; FP32 1e-4: six steps of 6e-8 roundings
of the vectors, amplified by at most |a| / b ~ 10 at each).
"""
import numpy as np
import pytest

from paper_1602_01863_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _recursion(apply, p, m):
    a, b = [], [0.0]
    v, prev = p / np.linalg.norm(p), np.zeros_like(p)
    for i in range(m):
        w = apply(v)
        a.append(np.vdot(v, w).real)
        w = w - a[-1] * v - b[-1] * prev
        b.append(np.linalg.norm(w))
        prev, v = v, w / b[-1]
    return np.array(a), np.array(b)


@pytest.mark.parametrize("cgs2", [False, True])
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("nv,nc,n,nd", [(2, 2, 3, 1), (1, 3, 3, 3), (2, 3, 4, 2), (3, 3, 8, 2)])
def test_coefficients(nv, nc, n, nd, prec, cgs2):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_01863_gb300 import bse
    steps, p = 6, 0 if prec == "f64" else 1
    ctx = bse.Context(0, torch.cuda.current_stream().cuda_stream)
    model = synth.draw_model(77, nv, nc)
    co = ctx.bse_build_coarse(model, n, p)
    it = ctx.bse_interp_setup(co, nd, bse.SCHEME_M3, 1.0, p)
    dirs = synth.POL3[:2].copy()
    a, b, pn2, done, _ = ctx.bse_haydock_run([it], [2], dirs, steps, bse.USE_GRAPH | (bse.REORTH_CGS2 if cgs2 else 0))
    dt = torch.complex128 if p == 0 else torch.complex64
    start = torch.empty((2, it.N), dtype=dt, device="cuda")
    ctx.bse_dipoles(it, dirs, start.data_ptr())
    y = torch.empty((1, it.N), dtype=dt, device="cuda")

    def apply(v):
        x = torch.from_numpy(v[None]).cuda().to(dt)
        ctx.bse_apply_h(it, 1, x.data_ptr(), y.data_ptr())
        return y[0].cpu().numpy().astype(np.complex128)

    for ch in range(2):
        ra, rb = _recursion(apply, start[ch].cpu().numpy().astype(np.complex128), steps)
        tol = (1e-12 if p == 0 else 1e-4) * np.max(np.abs(ra))
        assert done[ch] == steps
        assert np.max(np.abs(a[ch] - ra)) <= tol
        assert np.max(np.abs(b[ch, 1:] - rb[1:])) <= tol
    it.free()
    co.free()
    ctx.close()
