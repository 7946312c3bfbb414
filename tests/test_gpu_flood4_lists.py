"""The 4D flood fill's window pass when its lists fill up on a regular lattice.

On nodes at powers of two the sites midway between the elements are ties in
exact numbers: the site pass settles no element, and a component with its tied
edge (5 sites a side at stride 4) asks for more (site, neighbour) comparisons in
its sixth wave than the window pass lists (1152 against 1024).  The elements then
leave the window pass for the whole-lattice fill, and with more of them than it
has blocks, a block takes several, one after the other.
"""
import numpy as np
import pytest

import oracle.oracle4d as Q
from paper_1705_03750_gb300 import inputs4d as I4

pytestmark = pytest.mark.gpu


# fewer elements than the window pass has blocks, and more
@pytest.mark.parametrize("n,blocks_take_several", [((9, 9, 13, 9), False), ((13, 13, 13, 27), True)])
def test_elements_whose_comparisons_outgrow_their_list(n, blocks_take_several):
    from paper_1705_03750_gb300 import vlamet4d as V4
    half = [(a - 1) / 16 for a in n]
    rc = I4.HALOS4D_16.with_(n=n, s=4, lo=tuple(-h for h in half), hi=tuple(half))
    g = V4.Solver4D(V4.config(rc, pad=8))
    o = Q.Oracle4D.from_run(rc, pad=8)
    f0 = I4.initial_f4(rc)
    g.set_f(f0)
    o.set_f(f0)
    el = o.elements()      # the lattice of the reset
    g.step(1)              # (right after a reset the map is flooded as a whole, a block per element)
    o.step(1)
    for _ in range(2):
        g.set_elements(el)
        o.set_elements(el)
        fo = o.reconstruct()
        g.reconstruct()
        g.sync()
        assert (g.read_map() == o.last_map()).all()
        assert np.abs(g.read_f() - fo).max() <= 1e-12 * np.abs(fo).max()
        over = g.map_stats()["window_overflows"]
        assert over > (152 * 16 if blocks_take_several else 0.8 * len(el))
