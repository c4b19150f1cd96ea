"""Near stencil in the common basis where its row pairs, row lists and grids end.

FP32 pairs target rows along the whole zone (odd L: the last pair has one row; odd
n_div: a pair may span two cells), small grids share the source rows of a target
between the warps of a block, wide regions loop over the offsets.  Compared with the
general kernels on the same overlaps, handed over by the caller.

Bars: FP64 1e-12 of max |y| (the oracle tests' bar); FP32 4e-5: each side's own bar
against the oracle is 2e-5 of max |y|.
"""
import numpy as np
import pytest

from oracle import interp as oi
from paper_1602_01863_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = [  # nv, nc, n, n_div, width, vectors
    (1, 1, 3, 1, 1.0, 1),      # L = 3: the smallest odd zone, 7 offsets
    (2, 2, 5, 1, 2.4, 3),      # odd zone without subdivision, the other cell per row
    (2, 3, 3, 3, 1.0, 2),      # L = 9: pairs span cells, the last row alone; shared rows
    (3, 3, 7, 3, 1.0, 4),      # the same with runs of cells
    (2, 2, 3, 5, 1.2, 2),      # odd n_div with two z blocks, L = 15, R = 6
    (1, 2, 7, 2, 3.2, 2),      # R = 6 for n_div 2: the loop over offsets
    (2, 1, 4, 2, 0.5, 1),      # 7 offsets, fewer source rows than are worth sharing
    (4, 4, 5, 4, 1.5, 1),      # R = 6, runs of four cells and one
]


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "-".join(map(str, s)))
def test_near_rows(shape, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_01863_gb300 import bse
    nv, nc, n, nd, width, nvec = shape
    p = 0 if prec == "f64" else 1
    m = synth.draw_model(43, nv, nc)
    I = oi.Interp(m, n, nd, width=width, build_dense_kc=False)
    ctx = bse.Context(0, torch.cuda.current_stream().cuda_stream)
    out = []
    for scheme, dense in ((bse.SCHEME_M3, None), (bse.SCHEME_M3 | bse.NF_CUDA_CORES, {"Dv": I.Dv, "Dc": I.Dc})):
        co = ctx.bse_build_coarse(m, n, p)
        it = ctx.bse_interp_setup(co, nd, scheme, width, p, dense)
        x = torch.from_numpy(synth.random_vectors(19, (nvec, it.N))).cuda().to(torch.complex128 if p == 0 else torch.complex64)
        y = torch.empty_like(x)
        ctx.bse_apply_h(it, nvec, x.data_ptr(), y.data_ptr())
        out.append(y.cpu().numpy().astype(np.complex128))
        it.free()
        co.free()
    ctx.close()
    assert np.max(np.abs(out[0] - out[1])) <= (1e-12 if p == 0 else 4e-5) * np.max(np.abs(out[1]))
