"""The FP64 path's fixed-point values against the oracle.

The reconstruction and the remap evaluate offsets in units of 2^-52 cells and
node values in units of 2^-59 of the largest of a stencil; both sides are
therefore apart by the oracle's own FP64 rounding: an index position of up to
n cells carries a few units of n 2^-53, which changes f by at most that times
the largest difference of neighbouring nodes, plus some twenty roundings of
the sum: (8 n + 32) 2^-53 max|f| (max|f| bounds the differences here).
"""
import numpy as np
import pytest

import oracle.oracle as O
from paper_1705_03750_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1705_03750_gb300 import build as B  # noqa: E402

B.build()
from paper_1705_03750_gb300 import vlamet as V  # noqa: E402


# strides the remap's formats hold (2 to 64) and one each side; odd and even
# sides (lattice positions on nodes and between them); a sheared state whose
# elements lie more than the records' 32 sites from some of theirs
@pytest.mark.parametrize("nx,nv,s,shear,curve", [
    (64, 64, 4, 0.0, 0.0), (65, 47, 4, 0.1, 0.0), (48, 51, 1, 0.05, 0.0), (50, 49, 2, 0.1, 0.02),
    (131, 96, 3, 0.2, 0.05), (200, 150, 8, 0.3, 0.02), (260, 200, 64, 0.1, 0.01), (300, 280, 65, 0.1, 0.0),
    (90, 300, 8, 1.5, 0.0), (96, 96, 8, 0.1, 0.4),
    # from 2^15 sites on the values are formed in fixed point, below in FP64
    (181, 181, 4, 0.1, 0.0), (182, 181, 4, 0.1, 0.02), (210, 190, 1, 0.05, 0.0), (255, 180, 2, 0.2, 0.02),
    (190, 260, 8, 1.5, 0.0), (200, 200, 8, 0.1, 0.4)])
@pytest.mark.parametrize("scale", [1.0, 1e-290, 1e300])
def test_values_match_the_oracle(nx, nv, s, shear, curve, scale):
    rc = I.SPITZER_128.with_(nx=nx, nv=nv, s=s, G=0.0)
    f0 = I.initial_f(rc) * scale
    g = V.Solver(V.Config.from_run(rc))
    o = O.Oracle(nx, nv, rc.x_lo, rc.x_hi, rc.v_lo, rc.v_hi, s, rc.dt, rc.n_s, rc.G)
    g.set_f(f0)
    o.set_f(f0)
    el = o.elements().copy()
    el[:, 0] += shear * el[:, 1]
    el[:, 3] += shear
    # small smooth second-order terms, consistent in sign between neighbours
    el[:, 6:9] += curve * np.sin(2.0 * el[:, :1]) * np.array([1.0, 0.3, 0.2])
    el[:, 9:12] += curve * np.cos(1.5 * el[:, 1:2]) * np.array([0.4, -0.2, 0.5])
    o.set_elements(el)
    g.set_elements(np.ascontiguousarray(el.T))
    g.reconstruct()
    fo = o.reconstruct()
    tol = (8 * max(nx, nv) + 32) * 2.0 ** -53 * np.abs(f0).max()
    assert np.abs(g.read_f() - fo).max() <= tol
    eta = g.read_eta()
    assert np.abs(eta - o.eta()).max() <= 1e-13 * np.abs(eta).max()
    fr, _ = o.remap_resample()
    g.remap()
    assert np.abs(g.read_fini() - fr).max() <= 2 * tol  # the blend adds its quotient's roundings
