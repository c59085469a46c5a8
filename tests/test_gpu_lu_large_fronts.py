"""jac_reduced_solve on fronts far beyond what a cluster of CTAs holds: complete
graphs, one front of all their unknowns, and complete graphs that share buses.
Checks and tolerances of test_gpu_lu_fronts.
"""
import numpy as np
import pytest

from gridcases import make_grid
import test_gpu_lu_fronts as fronts

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1201, 1202])
def test_one_front_above_1200_unknowns(n):
    """Every pivot block, not only those that fit shared memory."""
    fronts.test_one_front(n)


@pytest.mark.parametrize("n", [257, 286, 287, 288, 289, 319, 321, 384, 385])
def test_one_front_at_the_edges_of_panels(n):
    """Panels of 32 pivots, tiles of 64."""
    fronts.test_one_front(n)


@pytest.mark.parametrize("own,shared", [(100, 31), (112, 32), (129, 17), (145, 48), (96, 65)])
def test_large_front_below_a_large_front(own, shared):
    """Three complete graphs, the later ones joined to the first by `shared` of its
    buses: large fronts of 2 own pivots and borders about the tiles' edges, whose updates
    reach a large root."""
    rng = np.random.default_rng(own)
    core = list(range(140))
    br, nb = fronts._clique(core, rng), len(core)
    for k in range(2):
        at = core[1 + 9 * k:1 + 9 * k + shared]
        new = list(range(nb, nb + own))
        nb += own
        br += [e for e in fronts._clique(at + new, rng) if not (e[0] in at and e[1] in at)]
    bt = np.ones(nb, np.int32)
    bt[0] = 3
    bt[5::7] = 2
    fronts._check(make_grid(nb, br), bt)


@pytest.mark.parametrize("core,own,shared", [(3, 150, 2), (9, 140, 1), (40, 131, 5)])
def test_small_fronts_above_a_large_front(core, own, shared):
    """A large front whose border reaches small ones: its ancestors are of its class,
    with panels of a few pivots."""
    rng = np.random.default_rng(own)
    br = fronts._clique(list(range(core)), rng)
    new = list(range(core, core + own))
    at = list(range(shared))
    br += [e for e in fronts._clique(at + new, rng) if not (e[0] in at and e[1] in at)]
    nb = core + own
    for k in range(5):   # a chain of small cliques off the core
        ring = list(range(nb, nb + 4))
        nb += 4
        br += fronts._clique([core - 1 - k % core] + ring, rng)
    bt = np.ones(nb, np.int32)
    bt[nb - 1] = 3
    fronts._check(make_grid(nb, br), bt)
