"""Set-up of systems with few bands: tiles of K_c and warps of the dense tables hold as many points as fit.

K_c against the oracle (1e-13 of max |K|, the bar of the other K_c tests) where tiles of
55, 32, 21, 16, 12 and 9 points end, and the time of bse_build_coarse for 1x1 bands
against 2x2 bands of nearly the same dimension: the work per entry is the
same but for the smaller tiles and the padding of the last ones, so three times
as long is too long.
"""
import time

import numpy as np
import pytest

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


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nv,nc,n", [(1, 1, 4), (1, 1, 5), (2, 1, 4), (1, 3, 3), (2, 2, 4), (1, 5, 3), (7, 1, 3)])
def test_kc_of_few_bands(ctx, nv, nc, n, prec):
    m = synth.draw_model(56, nv, nc)
    co = ctx.bse_build_coarse(m, n, prec)
    K = co.get_kc()
    ref = om.kernel_matrix(om.GridModel(m, om.coarse_coords(n), n))
    assert np.max(np.abs(K - ref)) <= (1e-13 if prec == 0 else 2.0 ** -23) * np.max(np.abs(ref))
    assert np.array_equal(K, K.conj().T)
    co.free()


def _median_ms(f):
    t = []
    for _ in range(6):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        h = f()
        t.append(1e3 * (time.perf_counter() - t0))
        h.free()
    return float(np.median(t[1:]))


def test_time_of_kc_with_one_band_pair(ctx):
    one, four = synth.draw_model(57, 1, 1), synth.draw_model(57, 2, 2)
    t1 = _median_ms(lambda: ctx.bse_build_coarse(one, 16, 1))         # N_c = 4096
    t4 = _median_ms(lambda: ctx.bse_build_coarse(four, 10, 1))        # N_c = 4000
    print(f"K_c, 1x1 bands {t1:.2f} ms, 2x2 bands {t4:.2f} ms")
    assert t1 <= 3 * t4


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nv,nc,n,nd", [(1, 1, 3, 3), (1, 1, 2, 5), (1, 2, 3, 3), (2, 2, 3, 2), (2, 1, 2, 3), (1, 3, 2, 3), (3, 2, 3, 2), (8, 8, 2, 2)])
def test_dense_tables_of_few_bands(ctx, nv, nc, n, nd, prec):
    """Dipoles, and H with overlaps formed by set-up: the last warp's points, one to sixteen to a warp.

    The dipoles are FP64 sums rounded once to the vector precision.  H: 1e-12 of max |H x| in FP64, 2e-5 in FP32,
    the bars of the H application tests.  Generators that are not Hermitian keep the overlap tables."""
    from oracle import interp as oi
    from paper_1602_01863_gb300 import bse
    for hermitian in (True, False):
        m = synth.draw_model(58, nv, nc)
        if not hermitian:
            m.gen_v[0, 0, 0, 0] += 0.05j
        I = oi.Interp(m, n, nd, width=0.4)
        co = ctx.bse_build_coarse(m, n, prec)
        it = ctx.bse_interp_setup(co, nd, bse.SCHEME_M3, 0.4, prec)
        dt = torch.complex128 if prec == 0 else torch.complex64
        P = torch.empty((3, it.N), dtype=dt, device="cuda")
        ctx.bse_dipoles(it, np.eye(3), P.data_ptr())
        ref = np.stack([I.dipole(e) for e in np.eye(3)])
        assert np.max(np.abs(P.cpu().numpy() - ref)) <= (1e-13 if prec == 0 else 2.0 ** -23) * np.max(np.abs(ref))
        x = torch.from_numpy(synth.random_vectors(8, (2, it.N))).cuda().to(dt)
        y = torch.empty_like(x)
        ctx.bse_apply_h(it, 2, x.data_ptr(), y.data_ptr())
        yr = (I.H_dense("m3") @ x.cpu().numpy().astype(np.complex128).T).T
        assert np.max(np.abs(y.cpu().numpy() - yr)) <= (1e-12 if prec == 0 else 2e-5) * np.max(np.abs(yr))
        it.free()
        co.free()


def test_time_of_dense_tables_with_one_band_pair(ctx):
    """A point of 1x1 bands is a quarter of the work of one of 2x2 bands and has a quarter of the lanes, so its
    tables take well below the time of theirs (a warp to each point: 0.85 of it)."""
    from paper_1602_01863_gb300 import bse
    t = []
    for nb in (1, 2):
        co = ctx.bse_build_coarse(synth.draw_model(59, nb, nb), 8, 1)
        t.append(_median_ms(lambda: ctx.bse_interp_setup(co, 8, bse.SCHEME_M1, 1.0, 1)))
        co.free()
    print(f"set-up of 262144 points, 1x1 bands {t[0]:.2f} ms, 2x2 bands {t[1]:.2f} ms")
    assert t[0] <= 0.7 * t[1]
