"""K_c is Hermitian with its diagonal, and complex128 keeps small imaginary parts.

The diagonal of a Hermitian matrix is real, so the stored one is, exactly.
With real form factors up to imaginary parts of 1e-8 and an identity gauge, Im K_c
is a sum of products of size 1e-8.  Summed as such it is off by a few roundings
of those products: bar 1e-13 of its largest entry (26 harmonics, 7 terms each, below
100 roundings of 1.1e-16, times the ratio of a sum's terms to the largest sum).  A
difference of sums of size 1 would be off by 1e-16 / 1e-8.
"""
import numpy as np
import pytest

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


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("nv,nc,n", [(1, 1, 3), (1, 2, 1), (3, 3, 3), (5, 5, 2), (8, 8, 2)])
def test_hermitian_with_its_diagonal(ctx, nv, nc, n, prec):
    co = ctx.bse_build_coarse(synth.draw_model(54, nv, nc), n, prec)
    K = co.get_kc()
    assert np.any(K.imag)
    assert np.array_equal(K, K.conj().T)
    co.free()


@pytest.mark.parametrize("nv,nc,n", [(1, 2, 4), (3, 3, 3), (4, 6, 2)])
def test_small_imaginary_parts(ctx, nv, nc, n):
    m = synth.draw_model(55, nv, nc)
    m.gen_v[:] = 0.0
    m.gen_c[:] = 0.0
    m.mu[:] = m.mu.real + 1e-8j * m.mu.imag
    co = ctx.bse_build_coarse(m, n, 0)
    K = co.get_kc()
    # M(k, G) and Im K_c = pref 2 sum_G v(G) (M_r M'_i - M_i M'_r) in extended precision
    k = np.stack(np.meshgrid(*(np.arange(n),) * 3, indexing="ij"), -1).reshape(-1, 3).astype(np.longdouble) / n
    two_pi = np.longdouble(8) * np.arctan(np.longdouble(1))
    c, s = np.cos(two_pi * k), np.sin(two_pi * k)
    h = np.stack([np.ones_like(c[:, 0]), c[:, 0], s[:, 0], c[:, 1], s[:, 1], c[:, 2], s[:, 2]], 1)
    t = nv * nc
    mu = m.mu.reshape(7, 26, t)
    re = np.einsum("ph,hgt->ptg", h, mu.real.astype(np.longdouble)).reshape(-1, 26)
    im = np.einsum("ph,hgt->ptg", h, mu.imag.astype(np.longdouble)).reshape(-1, 26)
    g = synth.gvectors_nonzero()
    v = np.longdouble(2) * two_pi / (g * g).sum(1)
    ref = np.longdouble(2 * m.e_k / n ** 3) * ((re * v) @ im.T - (im * v) @ re.T)
    assert np.max(np.abs(K.imag - ref)) <= 1e-13 * np.max(np.abs(ref))
    co.free()
