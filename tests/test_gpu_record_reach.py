"""Elements whose fixed-point record serves no site, against the oracle.

A record serves none where the map's terms leave its range: an element that is
not finite, or one sheared so strongly that even the sites next to its start
site are out of it.  A site whose value needs such an element, its start site
like any other, takes the FP64 evaluation.  The element is changed after a step
and a reconstruction, whose records are those of another state.

An element that is not finite owns no site beside finite ones (they pass at its
sites, and its distance is never the smaller one); the remap blends with it.
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

SHEARED = "sheared"    # linear terms beyond the range; on or close to a site's v, so that it keeps its start site


# 2D records are used from 2^15 sites on; linear terms of 750 (stride 8) end their range
@pytest.mark.parametrize("nx,nv,s", [(200, 170, 8), (231, 190, 4)])
@pytest.mark.parametrize("change", [SHEARED, np.nan, np.inf])
def test_2d_values_beside_an_element_without_a_record(nx, nv, s, change):
    rc = I.SPITZER_128.with_(nx=nx, nv=nv, s=s, n_s=50)
    f0 = I.initial_f(rc)
    g = V.Solver(V.Config.from_run(rc))
    o = O.Oracle(nx, nv, rc.x_lo, rc.x_hi, rc.v_lo, rc.v_hi, s, rc.dt, rc.n_s, rc.G)
    g.set_f(f0)
    o.set_f(f0)
    g.step(1)
    o.step(1)
    el = o.elements().copy()
    g.set_elements(np.ascontiguousarray(el.T))
    g.reconstruct()                       # every element has a record of this state
    m = (o.Lx // 2 - 2) * o.Lv + o.Lv // 2
    if change is SHEARED:
        j = round((el[m, 1] - rc.v_lo) / o.dv)
        el[m, 1] = rc.v_lo + j * o.dv
        el[m, 2:6] = [1.0, 4000.0, 0.0, 1.0]
    else:
        el[m, 7] = change
    o.set_elements(el)
    g.set_elements(np.ascontiguousarray(el.T))
    fo = o.reconstruct()
    owners, _ = o.compute_map()
    g.reconstruct()
    assert (g.read_map() == owners).all() and (owners == m).any() == (change is SHEARED)
    tol = (8 * max(nx, nv) + 32) * 2.0 ** -53 * np.abs(f0).max()
    assert np.abs(g.read_f() - fo).max() <= tol
    fr, _ = o.remap_resample()
    g.remap()
    assert np.abs(g.read_fini() - fr).max() <= 2 * tol


# 4D records end at linear terms of 60
@pytest.mark.parametrize("n,s", [((12, 10, 11, 12), 3), ((14, 13, 12, 13), 4)])
@pytest.mark.parametrize("change", [SHEARED, np.nan, np.inf])
def test_4d_values_beside_an_element_without_a_record(n, s, change):
    rc = I4.HALOS4D_16.with_(n=n, s=s, n_s=50)
    f0 = I4.initial_f4(rc)
    g = V4.Solver4D(V4.config(rc))
    o = Q.Oracle4D.from_run(rc)
    g.set_f(f0)
    o.set_f(f0)
    g.step(1)
    o.step(1)
    el = o.elements()
    g.set_elements(el)
    g.reconstruct()
    m = 0
    for a in range(4):
        m = m * o.Ldims[a] + o.Ldims[a] // 2
    if change is SHEARED:
        j = round((el[m, 2] - rc.lo[2]) / rc.d[2])
        el[m, 2] = rc.lo[2] + (j - 3e-4 * s) * rc.d[2]
        T = np.eye(4)
        T[0, 2] = 400.0
        el[m, 4:20] = T.ravel()
    else:
        el[m, 33] = change
    o.set_elements(el)
    g.set_elements(el)
    fo = o.reconstruct()
    owners = o.last_map()
    g.reconstruct()
    g.sync()
    assert (g.read_map() == owners).all() and (owners == m).any() == (change is SHEARED)
    assert np.abs(g.read_f() - fo).max() <= 1e-12 * np.abs(fo).max()
    fr, _ = o.remap_resample()
    g.remap()
    g.sync()
    assert np.abs(g.read_fini() - fr).max() <= 1e-12 * np.abs(fr).max()


# a second-order term that a served offset multiplies by little: 65 element
# spacings per spacing squared, 6 at two sites from the start at stride 8
@pytest.mark.parametrize("b", [40.0, 65.0])
def test_4d_values_of_an_element_with_a_strong_second_order_term(b):
    n, s = (17, 11, 19, 12), 8
    rc = I4.HALOS4D_16.with_(n=n, s=s, n_s=50)
    f0 = I4.initial_f4(rc)
    g = V4.Solver4D(V4.config(rc))
    o = Q.Oracle4D.from_run(rc)
    g.set_f(f0)
    o.set_f(f0)
    g.step(1)
    o.step(1)
    el = o.elements()
    m = 0
    for a in range(4):
        m = m * o.Ldims[a] + o.Ldims[a] // 2
    dm = s * np.array(rc.d)
    j = round((el[m, 2] - rc.lo[2]) / rc.d[2])
    el[m, 2] = rc.lo[2] + (j - 0.3) * rc.d[2]
    el[m, 4:20] = np.eye(4).ravel()
    el[m, 20:60] = 0.0
    el[m, 20 + 7] = -2.0 * b * dm[0] / dm[2] ** 2       # H_x,vx vx
    o.set_elements(el)
    g.set_elements(el)
    fo = o.reconstruct()
    owners = o.last_map()
    g.reconstruct()
    g.sync()
    assert (g.read_map() == owners).all() and (owners == m).any()
    assert np.abs(g.read_f() - fo).max() <= 1e-12 * np.abs(fo).max()
    fr, _ = o.remap_resample()
    g.remap()
    g.sync()
    assert np.abs(g.read_fini() - fr).max() <= 1e-12 * np.abs(fr).max()
