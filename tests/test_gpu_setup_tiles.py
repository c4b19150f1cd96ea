"""Set-up and pair-data kernels at the edges of their tiles.

K_c is computed in tiles of coarse points on and above the diagonal and mirrored:
band counts from 1x1 to 8x8 (tiles of 8 points down to 1), numbers of points that
leave a partial tile; 1e-13 of max |K| against the oracle, Hermitian off the diagonal.
Pair data with the overlaps formed from the gauge against the same overlaps given
by the caller (both round them to the vector precision, sums in FP32): 1e-4 of max |Y|,
the bar of the oracle test; features equal.
"""
import numpy as np
import pytest

from oracle import interp as oi
from oracle import model as om
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


@pytest.mark.parametrize("nv,nc,n", [(1, 1, 3), (1, 2, 1), (3, 3, 3), (5, 5, 2), (2, 7, 3), (8, 8, 2)])
def test_kc_tiles(ctx, nv, nc, n):
    m = synth.draw_model(51, nv, nc)
    co = ctx.bse_build_coarse(m, n, 0)
    K = co.get_kc()
    ref = om.kernel_matrix(om.GridModel(m, om.coarse_coords(n), n))
    assert np.max(np.abs(K - ref)) <= 1e-13 * np.max(np.abs(ref))
    off = K - K.conj().T
    np.fill_diagonal(off, 0)
    assert not np.any(off)
    co.free()


@pytest.mark.parametrize("nv,nc,n,nd,nb1,prec", [(1, 1, 3, 2, 0, 1), (8, 3, 2, 2, 0, 1), (3, 8, 2, 3, 1, 1), (4, 6, 2, 4, 0, 1),
                                                 (3, 5, 3, 2, 0, 0), (2, 2, 1, 2, 0, 0)])
def test_pairs_from_gauge_equal_pairs_from_tables(ctx, nv, nc, n, nd, nb1, prec):
    from paper_1602_01863_gb300 import bse
    m = synth.draw_model(52, nv, nc)
    I = oi.Interp(m, n, nd, build_dense_kc=False)
    rng = np.random.default_rng(4)
    kd, kd2 = rng.integers(0, I.Nk, 19), rng.integers(0, I.Nk, 19)
    out = []
    for dense in (None, {"Dv": I.Dv, "Dc": I.Dc}):
        co = ctx.bse_build_coarse(m, n, prec)
        it = ctx.bse_interp_setup(co, nd, bse.SCHEME_M1 | (bse.NB1 if nb1 else 0), 1.0, prec, dense)
        t = it.t
        X = torch.full((19 * t * t, 6 + 2 * t), float("nan"), device="cuda")
        Y = torch.full((19 * t * t, 2), float("nan"), device="cuda")
        ctx.bse_pairs_generate(it, kd, kd2, X.data_ptr(), Y.data_ptr())
        out.append((X.cpu().numpy(), Y.cpu().numpy()))
        it.free()
        co.free()
    (X, Y), (Xg, Yg) = out
    assert np.array_equal(X, Xg)
    assert np.max(np.abs(Y - Yg)) <= 1e-4 * np.max(np.abs(Yg))
