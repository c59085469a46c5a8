"""jac_reduced_solve at the edges of the column-block instances of the wide
fronts, and down a path of nested cliques whose fronts hand their x on.  Checks
and tolerances of test_gpu_lu_fronts.
"""
import numpy as np
import pytest

from gridcases import make_grid, series
import test_gpu_lu_fronts as fronts

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [65, 94, 95, 96, 97, 126])
def test_one_front_of_two_to_four_blocks(n):
    fronts.test_one_front(n)


@pytest.mark.parametrize("sizes", [(3, 4, 2, 5), (20, 9, 30, 3, 14), (90, 70, 3, 33, 2)])
def test_path_of_fronts(sizes):
    """Cliques in a row, each joined to half of the one before: the border of a
    front lies among the pivots and the border of its parent."""
    rng = np.random.default_rng(sum(sizes))
    br, nb, before = [], 0, []
    for m in sizes:
        new = list(range(nb, nb + m))
        nb += m
        br += fronts._clique(new, rng)
        br += [(x, new[i % m]) + series(0.01, 0.1) + (0.02, 1.0, 0.0)
               for i, x in enumerate(before[::2])]
        before = new + before[::4]
    bt = np.ones(nb, np.int32)
    bt[0] = 3
    bt[2::5] = 2
    fronts._check(make_grid(nb, br), bt)
