"""Set-up of systems with few bands: tiles of K_c hold as many coarse points as fit.

K_c against the oracle (1e-13 of max |K|, the bar of the other K_c tests) where tiles of
54, 32, 21, 16, 12 and 9 points end, and the time of bse_build_coarse for 1x1 bands
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
