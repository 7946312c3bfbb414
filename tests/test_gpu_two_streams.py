"""Two solvers stepping at once on two streams, each from its own thread.

A step holds a cooperative launch whose blocks wait for one another, between
kernels that are placed while the one before drains; two solvers' steps share the
chip.  Each gives what it gives alone, bit for bit.
"""
import threading

import numpy as np
import pytest

from paper_1705_03750_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1705_03750_gb300 import build as B  # noqa: E402

B.build()
from paper_1705_03750_gb300 import vlamet as V  # noqa: E402

RUNS = [(I.HALOS_4096.with_(nx=700, nv=520, n_s=10), V.VM_FP32_MIXED),
        (I.SPITZER_128.with_(nx=301, nv=217, s=8, n_s=10), V.VM_FP64)]


def solve(rc, prec, stream, out, at=None):
    dtype = np.float32 if prec == V.VM_FP32_MIXED else np.float64
    with torch.cuda.stream(stream):
        s = V.Solver(V.Config.from_run(rc, prec), stream=stream)
        s.set_f(I.initial_f(rc))
        s.sync()
        if at:
            at.wait()
        s.step(25)
        s.sync()
        out.append((s.read_f(dtype), s.read_fini(dtype), s.elements()))


def test_two_solvers_on_two_streams():
    alone = []
    for rc, prec in RUNS:
        solve(rc, prec, torch.cuda.Stream(), alone)
    for _ in range(3):
        at, outs = threading.Barrier(2), [[], []]
        threads = [threading.Thread(target=solve, args=(rc, prec, torch.cuda.Stream(), o, at))
                   for (rc, prec), o in zip(RUNS, outs)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        for o, a in zip(outs, alone):
            for x, y in zip(o[0], a):
                assert np.array_equal(x, y)
