"""H application in the common basis of the gauge against the general kernels.

With the model's tables the library factors the overlaps through U(k); with the
same overlaps handed over by the caller it runs the general kernels.  Both
compute the same H, so the two results are compared over band counts, meshes,
widths, weights, vector counts and precisions, where tiles, chunks and halos end.

Bars: FP64 1e-12 of max |y|, the bar of the oracle tests.  FP32 (the general
near field on the CUDA cores): each side's own bar against the oracle is 2e-5
of max |y|, so they differ by at most 4e-5.
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


def _apply(ctx, m, n, nd, scheme, width, kc, vec, nvec, dense=None):
    co = ctx.bse_build_coarse(m, n, kc)
    it = ctx.bse_interp_setup(co, nd, scheme, width, vec, dense)
    x = synth.random_vectors(17, (nvec, it.N))
    xt = torch.from_numpy(x).cuda().to(torch.complex128 if vec == 0 else torch.complex64)
    y = torch.empty_like(xt)
    ctx.bse_apply_h(it, nvec, xt.data_ptr(), y.data_ptr())
    again = torch.empty_like(xt)
    ctx.bse_apply_h(it, nvec, xt.data_ptr(), again.data_ptr())
    assert torch.equal(y, again)
    out, near = y.cpu().numpy().astype(np.complex128), it.n_near
    it.free()
    co.free()
    return x, out, near


SHAPES = [  # nv, nc, n, n_div, scheme, width, NB1, vectors
    (1, 1, 1, 4, 1, 0.4, 0, 1),      # one cell: every corner is the same point
    (1, 1, 7, 4, 1, 3.0, 0, 1),      # a box too wide for two FP32 source planes in shared memory
    (1, 2, 5, 4, 1, 2.2, 0, 2),      # the same in FP64
    (2, 1, 2, 3, 1, 0.9, 0, 4),      # two cells per axis, 16 columns used of 32
    (2, 3, 3, 1, 1, 1.0, 0, 3),      # no subdivision
    (3, 3, 3, 2, 1, 1.2, 1, 3),      # one-neighbour weights, odd mesh
    (3, 5, 5, 3, 1, 1.5, 0, 4),      # odd everything, 120 columns
    (2, 2, 4, 5, 1, 1.0, 0, 3),      # n_div above 4: two z blocks, a padded row
    (4, 4, 4, 4, 1, 1.0, 0, 3),
    (4, 6, 3, 4, 1, 1.4, 0, 1),
    (8, 8, 2, 2, 1, 0.9, 0, 2),      # the largest band counts
    (7, 5, 3, 2, 0, 1.0, 0, 3),      # Method 1
    (2, 2, 16, 2, 0, 1.0, 0, 1),     # more cells than dot partials
]


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "-".join(map(str, s)))
def test_common_basis_equals_general_kernels(ctx, shape, prec):
    from paper_1602_01863_gb300 import bse
    nv, nc, n, nd, scheme, width, nb1, nvec = shape
    kc, vec = {"f64": (0, 0), "f32": (1, 1), "bf16": (2, 1)}[prec]
    m = synth.draw_model(41, nv, nc)
    I = oi.Interp(m, n, nd, width=width, build_dense_kc=False)
    dense = {"Dv": I.Dv, "Dc": I.Dc}
    sch = scheme | (bse.NB1 if nb1 else 0)
    x, y, near = _apply(ctx, m, n, nd, sch, width, kc, vec, nvec)
    _, g, near_g = _apply(ctx, m, n, nd, sch | bse.NF_CUDA_CORES, width, kc, vec, nvec, dense)
    assert near == near_g
    assert np.max(np.abs(y - g)) <= (1e-12 if prec == "f64" else 4e-5) * np.max(np.abs(g))


def test_non_hermitian_generators_keep_the_general_path(ctx):
    """U(k) is not unitary then, so overlaps do not factor: 1e-12 against the oracle."""
    m = synth.draw_model(42, 2, 3)
    m.gen_v[0, 0, 0, 1] += 0.05
    x, y, _ = _apply(ctx, m, 3, 2, 1, 1.0, 0, 0, 1)
    ref = oi.Interp(m, 3, 2, width=1.0).H_dense("m3") @ x[0]
    assert np.max(np.abs(y[0] - ref)) <= 1e-12 * np.max(np.abs(ref))
