"""The remap's blend where every weight of a site is small, against the oracle.

Two neighbouring columns of elements are moved apart until the sites between
them lie at d = 1 - 5e-5 from both: the weights 2 (1 - d)^3 are 2e-13, and their
quotient is as exact as 1 - d.  The oracle's d carries a few units of n 2^-53 / s,
so its mean of two positions Delta cells apart errs by some 3 (4 n + 16) 2^-53 / s
/ (1 - d) Delta cells, and so does the FP64 evaluation here; f by that times its
largest change per cell (1.5 times the largest difference of neighbours).
"""
import numpy as np
import pytest

import oracle.oracle as O
import oracle.oracle4d as Q
from paper_1705_03750_gb300 import inputs as I
from paper_1705_03750_gb300 import inputs4d as I4

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1705_03750_gb300 import build as B  # noqa: E402

B.build()
from paper_1705_03750_gb300 import vlamet as V  # noqa: E402
from paper_1705_03750_gb300 import vlamet4d as V4  # noqa: E402

QX = 0.99925           # distance along x, in element spacings
ONE_LESS_D = 2.5e-4      # at least this with the offsets across x below


def tolerance(n, s, f, one_less_d=ONE_LESS_D):
    steps = max(np.abs(np.diff(f, axis=a)).max() for a in range(f.ndim))
    return 2 * 3 * (4 * n + 16) * 2.0 ** -53 / s / one_less_d * (2 * s) * 1.5 * steps


def test_2d_quotient_of_small_weights():
    nx, nv, s = 301, 121, 8
    rc = I.SPITZER_128.with_(nx=nx, nv=nv, s=s, G=0.0)
    f0 = I.initial_f(rc)
    g = V.Solver(V.Config.from_run(rc))
    o = O.Oracle(nx, nv, rc.x_lo, rc.x_hi, rc.v_lo, rc.v_hi, s, rc.dt, rc.n_s, rc.G)
    g.set_f(f0)
    o.set_f(f0)
    el = o.elements().copy()
    k = np.arange(o.ne) // o.Lv
    kc = o.Lx // 2 + 2
    # the site 8 cells beyond column kc - 1: QX from it, and from column kc
    el[k < kc, 0] += (8 - 8 * QX) * o.dx
    el[k >= kc, 0] += 8 * QX * o.dx
    el[:, 1] += 0.25 * o.dv
    d = np.hypot(QX, 0.25 / 8)
    assert ONE_LESS_D < 1 - d < 2 * ONE_LESS_D
    o.set_elements(el)
    g.set_elements(np.ascontiguousarray(el.T))
    fr, q = o.remap_resample()
    g.remap()
    tol = tolerance(max(nx, nv), s, f0) + 2 * (8 * max(nx, nv) + 32) * 2.0 ** -53 * np.abs(f0).max()
    assert np.abs(g.read_fini() - fr).max() <= tol


def test_4d_quotient_of_small_weights():
    n, s = (21, 9, 9, 9), 4
    rc = I4.HALOS4D_16.with_(n=n, s=s, G=0.0)
    f0 = I4.initial_f4(rc)
    g = V4.Solver4D(V4.config(rc))
    o = Q.Oracle4D.from_run(rc)
    g.set_f(f0)
    o.set_f(f0)
    el = o.elements()
    k = np.arange(o.ne) // (o.Ldims[1] * o.Ldims[2] * o.Ldims[3])
    kc = o.Ldims[0] // 2 + 1
    qx = (0.99997, 0.99996)     # (two different weights: their quotient of equal ones is exact)
    el[k < kc, 0] += (4 - 4 * qx[0]) * rc.d[0]
    el[k >= kc, 0] += 4 * qx[1] * rc.d[0]
    el[:, 1:4] += 0.01 * np.array(rc.d[1:])
    one_less_d = 2e-5
    assert all(one_less_d < 1 - np.sqrt(q ** 2 + 3 * 0.0025 ** 2) < 2 * one_less_d for q in qx)
    o.set_elements(el)
    g.set_elements(el)
    fr, _ = o.remap_resample()
    g.remap()
    g.sync()
    tol = tolerance(max(n), s, f0, one_less_d) + 1e-12 * np.abs(f0).max()
    assert np.abs(g.read_fini() - fr).max() <= tol
