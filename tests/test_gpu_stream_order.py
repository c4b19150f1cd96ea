"""Set-up, runs and training on a non-blocking stream while the default stream is busy.

Every copy and clear of the library has to be ordered with the kernels of the
context's stream by that stream alone.  Each call below is made while the
default stream still works through a queue of products, and has to give bit for bit
what a context with a stream of its own gives on an idle device.
"""
import numpy as np
import pytest

from oracle import interp as oi
from paper_1602_01863_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


class Busy:
    """Queues about 30 ms of products on the default stream."""

    def __init__(self):
        self.a = torch.randn((8192, 8192), device="cuda", dtype=torch.bfloat16)
        self.out = torch.empty_like(self.a)

    def __call__(self):
        for _ in range(50):
            torch.mm(self.a, self.a, out=self.out)


CASES = [  # K_c precision, vector precision, caller's overlaps, flags
    ("f64", 0, 0, False, 1),       # Gram-Schmidt with several blocks per vector: counters
    ("f32", 1, 1, False, 1),
    ("mixed", 2, 1, False, 0),     # counters of the update and of the tensor-core K_c apply
    ("caller", 2, 1, True, 0),     # lists and patterns of the general near field
]


def _recursion(stream, busy, kc, vec, caller, flags):
    from paper_1602_01863_gb300 import bse
    ctx = bse.Context(0, stream)
    m = synth.draw_model(91, 2, 2)
    n, nd = 5, 2                   # N = 4000: four blocks per vector
    dense = None
    if caller:
        I = oi.Interp(m, n, nd, build_dense_kc=False)
        dense = {"Dv": I.Dv, "Dc": I.Dc}
    busy()
    co = ctx.bse_build_coarse(m, n, kc)
    busy()
    it = ctx.bse_interp_setup(co, nd, bse.SCHEME_M3, 1.0, vec, dense)
    busy()
    a, b, pn2, steps, _ = ctx.bse_haydock_run([it], [2], synth.POL3[:2].copy(), 12, flags)
    it.free()
    co.free()
    ctx.close()
    return a, b, pn2, steps


@pytest.mark.parametrize("name,kc,vec,caller,flags", CASES, ids=[c[0] for c in CASES])
def test_recursion_beside_a_busy_default_stream(name, kc, vec, caller, flags):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    idle = _recursion(0, lambda: torch.cuda.synchronize(), kc, vec, caller, flags)
    side = torch.cuda.Stream()
    got = _recursion(side.cuda_stream, Busy(), kc, vec, caller, flags)
    torch.cuda.synchronize()
    for x, y in zip(idle, got):
        assert np.array_equal(x, y)


def _training(stream, busy, X, Y, p0):
    from paper_1602_01863_gb300 import bse
    ctx = bse.Context(0, stream)
    busy()
    mlp = ctx.bse_mlp_create(X.shape[1], len(X), p0)
    losses = []
    for _ in range(3):
        busy()
        losses.append(ctx.bse_mlp_train_step(mlp, len(X), X.data_ptr(), Y.data_ptr(), 1e-3))
    p = mlp.params()
    mlp.free()
    ctx.close()
    return np.array(losses), p


def test_training_beside_a_busy_default_stream():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_01863_gb300 import bse
    rng = np.random.default_rng(2)
    X = torch.from_numpy(rng.standard_normal((257, 14)).astype(np.float32)).cuda()
    Y = torch.from_numpy(rng.standard_normal((257, 2)).astype(np.float32)).cuda()
    p0 = (0.1 * rng.standard_normal(bse.load().bse_mlp_param_count(14))).astype(np.float32)
    idle = _training(0, lambda: torch.cuda.synchronize(), X, Y, p0)
    side, busy = torch.cuda.Stream(), Busy()
    torch.cuda.synchronize()
    got = _training(side.cuda_stream, busy, X, Y, p0)
    torch.cuda.synchronize()
    for x, y in zip(idle, got):
        assert np.array_equal(x, y)
