"""The influence map's site pass on strongly sheared states with exact ties.

A tile of sites and the ring of its neighbours have to propose the same owner for
a site.  On nodes at powers of two, sites midway between sheared elements are
equally close to two of them in exact numbers; far from an element (more than two
element spacings) the bounds of the FP32 evaluation have another form.  Owners
are whole numbers fixed by FP64 decisions in one order, so the map agrees exactly
with the oracle's and with that of the flood fill.
"""
import numpy as np
import pytest

import oracle.oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1705_03750_gb300 import build as B  # noqa: E402

B.build()
from paper_1705_03750_gb300 import vlamet as V  # noqa: E402


# x = a X + shear Y (+ an eighth-of-a-cell shift), v = b Y
@pytest.mark.parametrize("nx,nv,s,shear,a,b,shift", [
    (495, 108, 6, 3.5, 1.0, 0.875, (0.25, 0.125)), (234, 88, 5, -4.75, 1.25, 1.0, (0.0, 0.0)),
    (400, 120, 8, 6.0, 1.0, 1.0, (0.0, 0.0)), (301, 97, 4, -8.25, 0.75, 1.0, (0.0, 0.25))])
def test_map_of_sheared_ties(nx, nv, s, shear, a, b, shift):
    h = 1.0 / 64.0
    hi = ((nx - 1) * h, (nv - 1) * h)
    o = O.Oracle(nx, nv, 0.0, hi[0], 0.0, hi[1], s, 0.002, 100, 0.0)
    o.set_f(np.ones((nx, nv)))
    el = o.elements().copy()
    X, Y = el[:, 0] - 0.5 * hi[0], el[:, 1] - 0.5 * hi[1]
    el[:, 0] = 0.5 * hi[0] + a * X + shear * Y + shift[0] * h
    el[:, 1] = 0.5 * hi[1] + b * Y + shift[1] * h
    el[:, 2:6] = [a, shear, 0.0, b]
    o.set_elements(el)
    mo, _ = o.compute_map()
    for windows in (0, 1):
        g = V.Solver(V.Config(nx, nv, 0.0, hi[0], 0.0, hi[1], s, 0.002, 100, 0.0, V.VM_FP32_MIXED, map_windows=windows))
        g.set_f(np.ones((nx, nv)))
        g.set_elements(np.ascontiguousarray(el.T))
        for _ in range(2):       # the first map of a fresh lattice may go to the fill as a whole
            g.compute_map()
            assert (g.read_map() == mo).all()
