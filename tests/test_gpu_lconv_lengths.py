"""The learned convolution's line transforms over mesh sizes: every factor pair of the
in-register DFTs (1 to 8 points), lengths without one (the separate passes), transition
counts off the 4-entry blocks, 1 to 4 vectors, both vector precisions.

The reference is the stencil of the same network read back from the library (H applied
with and without the correction to unit vectors at one point gives its columns), applied
as a direct periodic sum in FP64 to a random vector: FP32 transforms of at most 33^3
points, 2e-5 of the largest entry of the correction (their error grows with log L),
plus the roundings of the two H x whose difference the correction is read from
(|H x| <= 5 |x| here, 2^-24 each, FP32 sums of a few terms: 2e-6 |x|).
"""
import numpy as np
import pytest

from paper_1602_01863_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,nd,nv,nc,nvec,prec", [
    (2, 2, 1, 1, 1, 1), (5, 1, 1, 2, 2, 1), (3, 2, 1, 3, 3, 1), (7, 1, 2, 1, 4, 1), (4, 2, 1, 1, 1, 0), (5, 2, 1, 2, 2, 1),
    (4, 3, 1, 1, 3, 1), (7, 2, 1, 1, 1, 1), (5, 3, 1, 1, 1, 0), (5, 4, 1, 1, 2, 1), (7, 3, 1, 1, 1, 1), (8, 3, 1, 1, 1, 1),
    (10, 3, 1, 1, 1, 1), (11, 1, 1, 2, 2, 1), (11, 3, 1, 1, 1, 1), (4, 2, 8, 8, 4, 1)])
def test_convolution_over_lengths(n, nd, nv, nc, nvec, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_01863_gb300 import bse
    ctx = bse.Context(0, torch.cuda.current_stream().cuda_stream)
    m = synth.draw_model(61, nv, nc)
    co = ctx.bse_build_coarse(m, n, prec)
    it = ctx.bse_interp_setup(co, nd, bse.SCHEME_M1, 1.0, prec)
    t, L = it.t, n * nd
    r = np.random.default_rng(3)
    mlp = ctx.bse_mlp_create(6 + 2 * t, 4096, (0.3 * r.standard_normal(ctx.lib.bse_mlp_param_count(6 + 2 * t))).astype(np.float32))
    radius = max(1, min(2, L // 2))
    dt = torch.complex128 if prec == 0 else torch.complex64

    def correction(x):
        """H x with the correction minus H x without it, for up to four vectors at a time."""
        out = []
        for i in range(0, len(x), 4):
            xt = torch.from_numpy(x[i:i + 4]).cuda().to(dt).contiguous()
            y0, y1 = torch.empty_like(xt), torch.empty_like(xt)
            ctx.bse_interp_set_learned(it, None, 0)
            ctx.bse_apply_h(it, len(xt), xt.data_ptr(), y0.data_ptr())
            ctx.bse_interp_set_learned(it, mlp, radius)
            ctx.bse_apply_h(it, len(xt), xt.data_ptr(), y1.data_ptr())
            out.append((y1 - y0).cpu().numpy().astype(np.complex128))
        return np.concatenate(out)

    cols = range(t) if t <= 4 else r.choice(t, 3, replace=False)          # transitions of the unit vectors
    unit = np.zeros((len(cols), it.N), dtype=np.complex128)
    for i, e in enumerate(cols):
        unit[i, e] = 1.0                                                    # at dense point 0
    T = correction(unit).reshape(len(cols), -1, t)                          # T(delta)[e1][e2] for e2 in cols
    cell = np.stack(np.meshgrid(*(np.arange(n),) * 3, indexing="ij"), -1).reshape(-1, 3)
    sub = np.stack(np.meshgrid(*(np.arange(nd),) * 3, indexing="ij"), -1).reshape(-1, 3)
    g = (cell[:, None] * nd + sub[None]).reshape(-1, 3)
    lin = np.empty((L, L, L), dtype=np.int64)
    lin[g[:, 0], g[:, 1], g[:, 2]] = np.arange(len(g))
    x = np.zeros((nvec, len(g), t), dtype=np.complex128)
    x[:, :, list(cols)] = synth.random_vectors(7, (nvec, len(g), len(cols)))
    ref = np.zeros_like(x)
    offs = [o for o in np.ndindex(L, L, L) if sum(min(v, L - v) ** 2 for v in o) < radius * radius]
    for o in offs:
        src = lin[tuple(np.mod(g - np.array(o), L).T)]
        ref += np.einsum("ce,pkc->pke", T[:, lin[o]], x[:, src][:, :, list(cols)])
    y = correction(x.reshape(nvec, -1)).reshape(ref.shape)
    assert np.max(np.abs(y - ref)) <= 2e-5 * np.max(np.abs(ref)) + 2e-6 * np.max(np.abs(x))
    it.free()
    co.free()
    mlp.free()
    ctx.close()
