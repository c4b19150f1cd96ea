"""Contexts of several threads at once, each with systems of a size of its own.

Kernels share their limits of shared memory between all of them, and the first
launches meet.  In a process of its own (fresh limits), eight threads set up
systems whose kernels need from little to much, start their first applications together,
and repeat; each has to get what a thread alone gets.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
import sys, threading
import numpy as np, torch
from paper_1602_01863_gb300 import bse, synth
torch.cuda.set_device(0)
SHAPES = [(1, 1, 3, 2, 0), (2, 2, 3, 2, 1), (3, 3, 4, 2, 1), (4, 4, 3, 3, 0), (4, 6, 3, 2, 1), (5, 5, 2, 4, 0), (6, 6, 2, 3, 1), (8, 8, 2, 2, 0)]
errors, results = [], [None] * len(SHAPES)

def work(i, meet):
    try:
        nv, nc, n, nd, scheme = SHAPES[i]
        stream = torch.cuda.Stream()
        ctx = bse.Context(0, stream.cuda_stream)
        m = synth.draw_model(70 + i, nv, nc)
        out = []
        if meet: meet.wait()
        for prec in (0, 1):
            co = ctx.bse_build_coarse(m, n, prec)
            it = ctx.bse_interp_setup(co, nd, scheme, 0.9, prec)
            with torch.cuda.stream(stream):
                x = torch.from_numpy(synth.random_vectors(i, (3, it.N))).cuda().to(torch.complex128 if prec == 0 else torch.complex64)
                y = torch.empty_like(x)
            stream.synchronize()
            mlp = None
            if scheme == 0:
                d_in = 6 + 2 * it.t
                p = (0.2 * np.random.default_rng(i).standard_normal(ctx.lib.bse_mlp_param_count(d_in))).astype(np.float32)
                mlp = ctx.bse_mlp_create(d_in, 2048, p)
                ctx.bse_interp_set_learned(it, mlp, 2)
            if meet: meet.wait()
            for _ in range(5):
                ctx.bse_apply_h(it, 3, x.data_ptr(), y.data_ptr())
            a, b, pn2, st, _ = ctx.bse_haydock_run([it], [2], synth.POL3[:2].copy(), 6, bse.USE_GRAPH)
            out += [y.cpu().numpy(), a, b]
            if mlp: mlp.free()
            it.free(); co.free()
        ctx.close()
        if results[i] is None: results[i] = out
        elif not all(np.array_equal(p, q) for p, q in zip(results[i], out)): errors.append((i, "differs"))
    except Exception as e:
        errors.append((i, repr(e)))
        if meet: meet.abort()

meet = threading.Barrier(len(SHAPES))
for together in (True, False):
    threads = [threading.Thread(target=work, args=(i, meet if together else None)) for i in range(len(SHAPES))]
    for t in threads:
        t.start()
        if not together: t.join()
    for t in threads: t.join()
print(errors)
sys.exit(1 if errors else 0)
"""


def test_first_launches_of_eight_threads():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    env = dict(os.environ, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr[-2000:]
