"""The 4D influence map's site pass against the oracle: owners are whole numbers
fixed by FP64 decisions in one order, so both agree exactly.
"""
import numpy as np
import pytest

import oracle.oracle4d as Q
from paper_1705_03750_gb300 import inputs4d as I4

pytestmark = pytest.mark.gpu


def _bent(el, rc, shear, curve, kick, seed):
    """x sheared along v, smooth second-order terms, and a few elements moved by
    up to a cell (their neighbours' components then overlap theirs or leave gaps)."""
    el = el.copy()
    el[:, 0:2] += shear * el[:, 2:4]
    T = np.eye(4)
    T[0, 2] = T[1, 3] = shear
    el[:, 4:20] = T.ravel()
    el[:, 20:60] = curve * np.sin(3.0 * el[:, :1] + np.arange(40))
    rng = np.random.default_rng(seed)
    m = rng.choice(len(el), max(1, len(el) // 40), replace=False)
    el[m, :4] += kick * rng.uniform(-1.0, 1.0, (len(m), 4)) * np.array(rc.d) * rc.s
    return el


# padded sides (side + 2 s) on the edges of the 2 x 4 x 4 x 8 tiles and beside
# them, odd and even (sites between the elements or midway), strides 1 to 8
@pytest.mark.parametrize("n,s,shear,curve,kick", [
    ((8, 12, 8, 8), 4, 0.0, 0.0, 0.0), ((9, 11, 13, 15), 4, 0.1, 0.0, 0.0), ((14, 18, 12, 16), 4, 0.3, 0.05, 0.0),
    ((13, 10, 11, 12), 3, 0.2, 0.02, 0.5), ((6, 7, 5, 9), 1, 0.1, 0.0, 0.3), ((12, 9, 10, 14), 2, 0.5, 0.1, 0.0),
    ((20, 17, 18, 19), 8, 0.2, 0.05, 0.5), ((4, 4, 4, 4), 1, 0.0, 0.0, 0.0), ((300, 4, 4, 5), 1, 0.1, 0.0, 0.0)])
@pytest.mark.parametrize("after_a_step", [False, True])
def test_map_equals_the_oracles(n, s, shear, curve, kick, after_a_step):
    from paper_1705_03750_gb300 import vlamet4d as V4
    rc = I4.HALOS4D_16.with_(n=n, s=s)
    g = V4.Solver4D(V4.config(rc))
    o = Q.Oracle4D.from_run(rc)
    f0 = I4.initial_f4(rc)
    g.set_f(f0)
    o.set_f(f0)
    el = _bent(o.elements(), rc, shear, curve, kick, sum(n))
    if after_a_step:       # (a map right after a reset is flooded where sites are midway)
        g.step(1)
        o.step(1)
    g.set_elements(el)
    o.set_elements(el)
    for _ in range(2):     # the second map finds the first one's arrays emptied
        fo = o.reconstruct()
        g.reconstruct()
        g.sync()
        assert (g.read_map() == o.last_map()).all()
    assert np.abs(g.read_f() - fo).max() <= 1e-12 * np.abs(fo).max()
    assert g.map_stats()["holes"] == o.map_stats()["holes"]


@pytest.mark.parametrize("word", [1, 9, 33])         # position, linear term, second-order term
@pytest.mark.parametrize("value", [np.nan, np.inf, 1e200])
def test_elements_that_are_not_finite_leave_the_others_to_the_fill(word, value):
    from paper_1705_03750_gb300 import vlamet4d as V4
    rc = I4.HALOS4D_16.with_(n=(12, 10, 11, 12), s=3)
    maps = []
    for step in (0, 1):    # flooded as a whole (sites midway, right after a reset); with the site pass
        g = V4.Solver4D(V4.config(rc))
        f0 = I4.initial_f4(rc)
        g.set_f(f0)
        el = g.elements()
        if step:
            g.step(1)
        el[[40, len(el) // 2], word] = value
        g.set_elements(el)
        g.reconstruct()
        g.sync()
        maps.append(g.read_map())
    assert np.array_equal(maps[0], maps[1])
