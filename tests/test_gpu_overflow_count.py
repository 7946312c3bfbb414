"""The number of elements whose component leaves the small windows.

It is a property of the components alone, so it is the same whether the site pass
settled an element or the flood fill claimed for it, and follows from the
components' extents in the oracle's percolation.
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


def expected(o, el, rc):
    """Elements whose component has a site on or beyond the edge of its window (32 x
    64 sites, 16 x 32 for an element with a neighbour missing) where the padded
    lattice goes on behind that edge."""
    box, n = o.component_bbox(), 0
    for m in range(o.ne):
        i_min, i_max, j_min, j_max = (int(b) for b in box[m])
        if i_min > i_max:
            continue
        k, l = divmod(m, o.Lv)
        h = 8 if k in (0, o.Lx - 1) or l in (0, o.Lv - 1) else 16
        i0 = int(np.floor((el[m, 0] - rc.x_lo) * (1.0 / o.dx) + 0.5))
        j0 = int(np.floor((el[m, 1] - rc.v_lo) * (1.0 / o.dv) + 0.5))
        n += ((i_min - i0 <= -h and i0 - h - 1 >= -rc.s) or (i_max - i0 >= h - 1 and i0 + h < rc.nx + rc.s) or
              (j_min - j0 <= -2 * h and j0 - 2 * h - 1 >= -rc.s) or (j_max - j0 >= 2 * h - 1 and j0 + 2 * h < rc.nv + rc.s))
    return n


# x = a X + shear Y, v = b Y: components beyond the windows along x, along v, and
# by their shear; the rim's alone; none
@pytest.mark.parametrize("nx,nv,s,shear,a,b,some", [
    (400, 300, 8, 0.0, 4.5, 1.0, True), (300, 400, 8, 0.1, 1.0, 9.0, True), (400, 300, 8, 1.5, 1.0, 1.0, True),
    (311, 207, 7, 0.3, 4.6, 2.2, True), (250, 250, 4, 0.05, 0.9, 0.9, True), (128, 100, 8, 0.0, 1.0, 1.0, False),
    (200, 260, 16, 0.0, 1.9, 1.0, True)])
def test_count_of_components_that_leave_the_small_windows(nx, nv, s, shear, a, b, some):
    rc = I.SPITZER_128.with_(nx=nx, nv=nv, s=s, G=0.0)
    f0 = I.initial_f(rc)
    o = O.Oracle(nx, nv, rc.x_lo, rc.x_hi, rc.v_lo, rc.v_hi, s, rc.dt, rc.n_s, rc.G)
    o.set_f(f0)
    el = o.elements().copy()
    x, v = el[:, 0].copy(), el[:, 1].copy()
    el[:, 0] = a * x + shear * v
    el[:, 1] = b * v
    el[:, 2:6] = [a, shear, 0.0, b]
    o.set_elements(el)
    mo, _ = o.compute_map()
    n = expected(o, el, rc)
    assert (n > 0) == some
    for windows in (0, 1):
        cfg = V.Config.from_run(rc)
        cfg.map_windows = windows
        g = V.Solver(cfg)
        g.set_f(f0)
        g.set_elements(np.ascontiguousarray(el.T))
        for _ in range(2):       # the first map of a fresh lattice may go to the fill as a whole
            g.compute_map()
            assert (g.read_map() == mo).all()
            assert g.diagnostics()["overflow_elements"] == n
