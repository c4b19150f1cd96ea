"""H with overlaps handed over by the caller: the general kernels, the tensor-core near field first.

With the model's overlaps the library works in the common basis; overlaps given by
the caller (here the model's own, from the oracle) keep the general kernels: restricted
pieces in FP16 with scales from the inputs' norms, the tensor-core near field beside
the K_c apply, and the staged FP32 kernels.

Bars: FP32 arithmetic 2e-5 of max |H x|; the tensor-core near field 5e-3 of max |near
field| of a row (11-bit operands, amplified about tenfold by the cancellation of y1
against h_head z).  Scaling an input by a power of two scales its pieces' factor
by the inverse, so the output scales exactly.

And the stencil of the common basis in FP32, weight by weight: H applied to unit vectors
against the same in FP64.  At a dense point the near part is one weight times two rotations
(2 (nv + nc) products each way) beside the interpolated part of at most 8 x 8 corner
products; with at most 64 roundings of 2^-24 of the parts' sizes there: 2^-18, and where the
corner products cancel, 16 roundings of the largest interpolated entry: 2^-20.
"""
import numpy as np
import pytest

from oracle import interp as oi
from paper_1602_01863_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_01863_gb300 import bse
    torch.cuda.set_device(0)
    c = bse.Context(0, torch.cuda.current_stream().cuda_stream)
    yield c
    c.close()


def _apply(ctx, it, x):
    xs = torch.from_numpy(np.ascontiguousarray(x)).cuda().to(torch.complex128 if it.vec_prec == 0 else torch.complex64)
    ys = torch.empty_like(xs)
    ctx.bse_apply_h(it, len(x), xs.data_ptr(), ys.data_ptr())
    return ys.cpu().numpy().astype(np.complex128)


def _handles(ctx, m, I, n, nd, scheme, kc, width=1.0):
    co = ctx.bse_build_coarse(m, n, kc)
    return co, ctx.bse_interp_setup(co, nd, scheme, width, 1, {"Dv": I.Dv, "Dc": I.Dc})


def _free(*handles):
    for h in handles:
        h.free()


@pytest.mark.parametrize("nv,nc,n,nd", [(4, 4, 3, 2), (3, 3, 3, 2), (2, 3, 3, 3), (1, 2, 3, 4), (3, 5, 3, 2)])
def test_tensor_core_near_field_whole_vector(ctx, nv, nc, n, nd):
    m = synth.draw_model(41, nv, nc)
    I = oi.Interp(m, n, nd, width=1.0)
    co, it = _handles(ctx, m, I, n, nd, 1, 1)
    H3, H1 = I.H_dense("m3"), I.H_dense("m1")
    x = synth.random_vectors(5, (3, it.N)).astype(np.complex64).astype(np.complex128)
    y, yr, nf = _apply(ctx, it, x), (H3 @ x.T).T, ((H3 - H1) @ x.T).T
    assert np.abs(y - yr).max() <= 2e-5 * np.abs(yr).max() + 5e-3 * np.abs(nf).max()
    assert np.abs(y - yr).max() > 1e-8 * np.abs(nf).max()          # FP16 operands: not the FP32 stencil
    _free(it, co)


def test_tensor_core_near_field_rows_and_wrap(ctx):
    """All sub-points of the first and the last coarse cell, whose partners wrap around the zone."""
    m, n, nd = synth.draw_model(43, 4, 4), 4, 4
    I = oi.Interp(m, n, nd, width=1.0, build_dense_kc=False)
    co3, it3 = _handles(ctx, m, I, n, nd, 1, 1)
    co1, it1 = _handles(ctx, m, I, n, nd, 0, 1)
    x = synth.random_vectors(6, (3, it3.N)).astype(np.complex64).astype(np.complex128)
    nf = _apply(ctx, it3, x) - _apply(ctx, it1, x)
    rows = np.concatenate([np.arange(nd ** 3), np.arange((n ** 3 - 1) * nd ** 3, n ** 3 * nd ** 3)])
    for v in (0, 2):
        ref, got = I.near_field_rows(x[v], rows), nf[v].reshape(I.Nk, I.t)[rows]
        assert np.max(np.abs(got - ref).max(axis=1) / np.abs(ref).max(axis=1)) <= 5e-3
    _free(it3, co3, it1, co1)


@pytest.mark.parametrize("kc", [1, 2])
@pytest.mark.parametrize("nv,nc,n,nd", [(3, 3, 4, 2), (4, 4, 4, 4), (2, 3, 5, 3)])
def test_scales_follow_each_vectors_norm(ctx, nv, nc, n, nd, kc):
    m = synth.draw_model(44, nv, nc)
    I = oi.Interp(m, n, nd, build_dense_kc=False)
    co, it = _handles(ctx, m, I, n, nd, 1, kc)
    x = synth.random_vectors(7, (3, it.N)).astype(np.complex64).astype(np.complex128)
    f = np.array([[1.0], [2.0 ** 20], [2.0 ** -30]])
    y, ys = _apply(ctx, it, x), _apply(ctx, it, f * x)
    assert np.all(np.isfinite(y)) and np.array_equal(ys, f * y)
    _free(it, co)


@pytest.mark.parametrize("nv,nc", [(3, 3), (4, 4), (4, 6), (2, 3)])
@pytest.mark.parametrize("scheme", [0, 1])
def test_staged_and_generic_kernels_in_fp32(ctx, nv, nc, scheme):
    """The FP32 kernels for 3x3, 4x4 and 4x6 bands, the generic ones for 2x3, near field on the CUDA cores."""
    from paper_1602_01863_gb300 import bse
    m, n, nd = synth.draw_model(13, nv, nc), 3, 2
    I = oi.Interp(m, n, nd, width=1.0)
    co, it = _handles(ctx, m, I, n, nd, scheme | bse.NF_CUDA_CORES, 1)
    x = synth.random_vectors(9, (3, it.N)).astype(np.complex64).astype(np.complex128)
    y, yr = _apply(ctx, it, x), (I.H_dense("m3" if scheme else "m1") @ x.T).T
    assert np.abs(y - yr).max() <= 2e-5 * np.abs(yr).max()
    _free(it, co)


def test_general_near_field_beside_the_kc_apply(ctx):
    """K_c apply and tensor-core near field side by side, in a graph and eagerly, and one after another: the same bits."""
    from paper_1602_01863_gb300 import bse
    m, n, nd = synth.draw_model(31, 4, 4), 5, 4
    I = oi.Interp(m, n, nd, build_dense_kc=False)
    co, it = _handles(ctx, m, I, n, nd, 1, 2)
    runs = [ctx.bse_haydock_run([it], [3], np.eye(3), 30, f) for f in (bse.USE_GRAPH, 0, bse.PROFILE, bse.USE_GRAPH)]
    assert np.all(np.isfinite(runs[0][0])) and np.all(runs[0][1][:, 1:] > 0)
    for r in runs[1:]:
        assert np.array_equal(r[0], runs[0][0]) and np.array_equal(r[1], runs[0][1])
    _free(it, co)


@pytest.mark.parametrize("nv,nc,n,nd,width", [(2, 3, 5, 4, 1.5), (3, 3, 7, 3, 1.0), (2, 2, 3, 5, 1.2), (1, 2, 7, 2, 3.2), (4, 4, 3, 2, 1.2), (1, 1, 4, 1, 1.9)])
def test_stencil_weights_in_fp32(ctx, nv, nc, n, nd, width):
    m = synth.draw_model(45, nv, nc)
    out = {}
    x = np.zeros((4, nv * nc * (n * nd) ** 3), dtype=np.complex128)
    at = np.random.default_rng(8).choice(x.shape[1], 4, replace=False)
    x[np.arange(4), at] = 1.0
    for prec in (0, 1):
        co = ctx.bse_build_coarse(m, n, prec)
        for scheme in (0, 1):
            it = ctx.bse_interp_setup(co, nd, scheme, width, prec)
            out[prec, scheme] = _apply(ctx, it, x).reshape(4, -1, nv * nc)
            _free(it)
        _free(co)
    near = np.abs(out[0, 1] - out[0, 0]).max(axis=2)
    m1 = np.abs(out[0, 0]).max(axis=2)
    other = np.where(m1 == m1.max(axis=1, keepdims=True), 0.0, m1).max()      # without the points' own energies
    bar = 2.0 ** -18 * (near + m1) + 2.0 ** -20 * other
    assert np.all(np.abs(out[1, 1] - out[0, 1]).max(axis=2) <= bar)
    if nd == 1:
        assert not np.any(near)                                    # every dense difference is a coarse one: the heads cancel
    else:
        assert np.count_nonzero(near > 1e-12 * near.max()) >= 4 * 7     # seven offsets and more were reached


@pytest.mark.parametrize("nv,nc,n,nd", [(3, 3, 4, 2), (2, 3, 5, 3)])
def test_zero_and_tiny_vectors(ctx, nv, nc, n, nd):
    """H 0 = 0 beside another vector, and a vector of norm 1e-18 keeps its scale."""
    m = synth.draw_model(46, nv, nc)
    I = oi.Interp(m, n, nd, build_dense_kc=False)
    co, it = _handles(ctx, m, I, n, nd, 1, 1)
    x = synth.random_vectors(12, (1, it.N)).astype(np.complex64).astype(np.complex128)
    y = _apply(ctx, it, np.concatenate([0 * x, x, 2.0 ** -66 * x]))
    assert not np.any(y[0])
    assert np.all(np.isfinite(y)) and np.array_equal(y[2], 2.0 ** -66 * y[1])
    _free(it, co)
