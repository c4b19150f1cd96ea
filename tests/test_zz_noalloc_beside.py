"""bse_apply_h_noalloc beside a Haydock run on the same handle.

The call shares nothing that either writes with the handle's other calls, so a
recursion in one thread (a context and stream of its own) and a loop of such calls in
another give bit for bit what each gives alone.
"""
import threading

import numpy as np
import pytest

from oracle import interp as oi
from paper_1602_01863_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("name,kc,vec,scheme,caller,shape", [
    ("m3-f64", 0, 0, 1, False, (3, 3, 4, 2, 2)), ("m3-mixed", 2, 1, 1, False, (3, 3, 4, 2, 2)),
    ("m1-f32", 1, 1, 0, False, (3, 3, 4, 2, 2)),
    ("caller-f32", 1, 1, 1, True, (3, 3, 4, 2, 2)), ("caller-mixed", 2, 1, 1, True, (3, 3, 4, 2, 2)),
    ("behind-the-rest", 1, 1, 1, False, (1, 1, 4, 2, 1)),     # columns of 32 take more than the pieces' place
    ("set-of-its-own", 0, 0, 1, False, (1, 1, 11, 4, 1)),     # and more than the array: 21.9 MB count, 27 MB follow
], ids=lambda v: v if isinstance(v, str) else "")
def test_noalloc_beside_a_recursion(name, kc, vec, scheme, caller, shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_01863_gb300 import bse
    nv, nc, n, nd, nvec = shape
    m = synth.draw_model(95, nv, nc)
    dense = None
    if caller:
        I = oi.Interp(m, n, nd, build_dense_kc=False)
        dense = {"Dv": I.Dv, "Dc": I.Dc}
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    run, other = (bse.Context(0, s.cuda_stream) for s in streams)
    co = run.bse_build_coarse(m, n, kc)
    it = run.bse_interp_setup(co, nd, scheme, 1.0, vec, dense)
    dirs = synth.POL3.copy()

    def recursion():
        return run.bse_haydock_run([it], [3], dirs, 60, bse.USE_GRAPH)[:3]

    dt = torch.complex128 if vec == 0 else torch.complex64
    # norms that differ by far, so that FP16 pieces need scales of their own
    x = (torch.from_numpy(synth.random_vectors(11, (nvec, it.N))) * torch.tensor([[1e3], [1e-4]])[:nvec]).cuda().to(dt)
    y = torch.empty_like(x)
    torch.cuda.synchronize()

    def apply():
        other.bse_apply_h_noalloc(it, nvec, x.data_ptr(), y.data_ptr())
        with torch.cuda.stream(streams[1]):
            return y.clone()

    ref_run, ref_y = recursion(), apply()
    own = torch.empty_like(x)
    run.bse_apply_h(it, nvec, x.data_ptr(), own.data_ptr())
    torch.cuda.synchronize()
    tol = 1e-12 if vec == 0 else 1e-5
    assert all(bool((p - q).abs().max() <= tol * p.abs().max()) for p, q in zip(own, ref_y))
    assert all(np.all(np.isfinite(v)) for v in ref_run) and bool(torch.isfinite(torch.view_as_real(ref_y)).all())
    got, done = [], threading.Event()

    def runs():
        try:
            for _ in range(6):
                got.append(recursion())
        finally:
            done.set()

    t = threading.Thread(target=runs)
    t.start()
    ys = [apply()]
    while not done.is_set():
        ys.append(apply())
    t.join()
    torch.cuda.synchronize()
    assert len(got) == 6 and len(ys) > 1
    for r in got:
        assert all(np.array_equal(p, q) for p, q in zip(r, ref_run))
    assert all(torch.equal(v, ref_y) for v in ys)
    it.free()
    co.free()
    run.close()
    other.close()
