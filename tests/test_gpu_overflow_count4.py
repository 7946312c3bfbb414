"""The 4D number of elements whose component outgrows the flood window is the same
whether the site pass settled an element or the flood fill claimed for it.

Right after a reset of a grid whose sites lie midway between its elements the map
is flooded as a whole; after a step the site pass runs.  The elements are set to
the same state for both: stretched along one axis, their components lines of a few
sites (the fill's lists hold every wave of them), on no tie.
"""
import numpy as np
import pytest

from paper_1705_03750_gb300 import inputs4d as I4

pytestmark = pytest.mark.gpu


# components short of the window's edge, on it, and beyond it
@pytest.mark.parametrize("n,s,axis,a,some", [
    ((14, 6, 6, 7), 1, 0, 2.0, False), ((14, 6, 6, 7), 1, 0, 4.0, True), ((6, 14, 6, 7), 1, 1, 7.0, True),
    ((6, 6, 14, 7), 1, 2, 4.5, True), ((24, 9, 9, 8), 2, 0, 4.5, True)])
def test_count_with_and_without_the_site_pass(n, s, axis, a, some):
    from paper_1705_03750_gb300 import vlamet4d as V4
    half = [(q - 1) / 16 for q in n]
    rc = I4.HALOS4D_16.with_(n=n, s=s, lo=tuple(-h for h in half), hi=tuple(half), n_s=50)
    f0 = I4.initial_f4(rc)
    seen = []
    for steps in (0, 1):
        g = V4.Solver4D(V4.config(rc))
        g.set_f(f0)
        el = np.array(g.elements())
        el[:, axis] *= a
        el[:, 4 + 5 * axis] = a
        el[:, :4] += 0.23 * np.array(rc.d)
        g.step(steps)
        g.set_elements(el)
        g.profile(True)
        g.reconstruct()
        g.sync()
        assert ("sites" in g.profile_read()) == (steps == 1)
        seen.append((g.read_map(), g.map_stats()["window_overflows"]))
    assert np.array_equal(seen[0][0], seen[1][0])
    assert seen[0][1] == seen[1][1] and (seen[0][1] > 0) == some
