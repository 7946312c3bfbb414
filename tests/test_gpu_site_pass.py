"""The influence map's site pass against the oracle and against the flood fill.

Owners are whole numbers fixed by FP64 decisions in one order, so all three
agree exactly.  map_windows=1 sends every element to the flood fill.
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


def bent(el, shear, curve, kick, seed):
    """Shear, smooth second-order terms, and a few elements moved by a cell or
    two (their neighbours' components then overlap theirs or leave gaps)."""
    el[:, 0] += shear * el[:, 1]
    el[:, 3] += shear
    el[:, 6:9] += curve * np.sin(2.0 * el[:, :1]) * np.array([1.0, 0.3, 0.2])
    el[:, 9:12] += curve * np.cos(1.5 * el[:, 1:2]) * np.array([0.4, -0.2, 0.5])
    rng = np.random.default_rng(seed)
    m = rng.choice(len(el), max(1, len(el) // 50), replace=False)
    el[m, :2] += kick * rng.uniform(-1.0, 1.0, (len(m), 2))
    return el


# padded sides (side + 2 s) of one tile of 32 x 64 sites, one less, one more and
# smaller than it; strides down to 1; sheared, curved and torn states; lattices
# at the longest the pass takes (4095 positions) and beyond it
@pytest.mark.parametrize("nx,nv,s,shear,curve,kick", [
    (24, 56, 4, 0.0, 0.0, 0.0), (23, 55, 4, 0.1, 0.0, 0.0), (25, 57, 4, 0.1, 0.02, 0.05), (56, 120, 4, 0.3, 0.05, 0.1),
    (87, 185, 4, 1.5, 0.0, 0.0), (30, 62, 1, 0.05, 0.0, 0.0), (31, 63, 1, 0.2, 0.05, 0.05), (61, 127, 2, 0.1, 0.02, 0.3),
    (4, 4, 1, 0.0, 0.0, 0.0), (5, 7, 2, 0.2, 0.0, 0.0), (131, 97, 3, 0.2, 0.4, 0.0), (200, 250, 16, 0.3, 0.2, 0.4),
    (300, 280, 65, 0.1, 0.05, 0.0), (375, 433, 8, 0.3, 0.05, 0.1), (600, 350, 7, 1.5, 0.02, 0.0), (16400, 8, 4, 0.0, 0.0, 0.0),
    (470, 497, 1, 0.05, 0.01, 0.05), (4080, 9, 1, 0.0, 0.0, 0.0), (4200, 9, 1, 0.0, 0.0, 0.0), (9, 4200, 1, 0.1, 0.0, 0.0)])
@pytest.mark.parametrize("f_th", [0.0, 1e-3])
def test_map_equals_the_oracles_and_the_flood_fills(nx, nv, s, shear, curve, kick, f_th):
    rc = I.SPITZER_128.with_(nx=nx, nv=nv, s=s, G=0.0)
    f0 = I.initial_f(rc)
    o = O.Oracle(nx, nv, rc.x_lo, rc.x_hi, rc.v_lo, rc.v_hi, s, rc.dt, rc.n_s, rc.G)
    if f_th:
        o.set_fth(f_th)
    o.set_f(f0)
    el = bent(o.elements().copy(), shear, curve, kick, nx * nv)
    o.set_elements(el)
    mo, st = o.compute_map()
    for windows in (0, 1):
        cfg = V.Config.from_run(rc)
        cfg.map_windows, cfg.f_th = windows, f_th
        g = V.Solver(cfg)
        g.set_f(f0)
        g.set_elements(np.ascontiguousarray(el.T))
        for _ in range(2):       # the first map of a fresh lattice may go to the fill as a whole
            g.compute_map()
            try:
                g.sync()
                assert st == 0
            except V.VlametError as e:
                assert e.status == st != 0
            mg = g.read_map()
            assert (mg == mo).all(), f"windows {windows}: {(mg != mo).sum()} sites differ"
        assert g.diagnostics()["holes"] == o.map_stats()["holes"]


@pytest.mark.parametrize("word", [0, 2, 7])          # position, linear term, second-order term
@pytest.mark.parametrize("value", [np.nan, np.inf, 1e200, -1e30])
def test_elements_that_are_not_finite_are_left_to_the_fill(word, value):
    rc = I.SPITZER_128.with_(nx=390, nv=370, s=4, G=0.0)
    f0 = I.initial_f(rc)
    maps = []
    for windows in (0, 1):
        cfg = V.Config.from_run(rc)
        cfg.map_windows = windows
        g = V.Solver(cfg)
        g.set_f(f0)
        el = np.array(g.elements())
        el[word, [7, el.shape[1] // 2, el.shape[1] // 2 + 40]] = value
        g.set_elements(np.ascontiguousarray(el))
        for _ in range(2):
            g.compute_map()
            try:
                g.sync()
            except V.VlametError as e:
                assert e.status == 4
            maps.append(g.read_map())
    for m in maps[1:]:
        assert np.array_equal(m, maps[0])
