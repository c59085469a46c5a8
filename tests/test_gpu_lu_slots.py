"""jac_reduced_solve where the last pivot rows of a cluster's front have no later
row behind them on some of its CTAs: fronts with fewer border unknowns than the
cluster has CTAs, roots, and batches of pivot rows that end with one to eight
rows.  Checks and tolerances of test_gpu_lu_fronts.
"""
import numpy as np
import pytest

from gridcases import make_grid
import test_gpu_lu_fronts as fronts

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [134, 137, 141, 201, 204, 208])
def test_root_past_a_batch_of_rows(n):
    """Batches of 133 rows below 192 unknowns, of 100 from there on."""
    fronts.test_one_front(n)


@pytest.mark.parametrize("buses", [36, 68, 101])
@pytest.mark.parametrize("shared", [1, 2, 3, 4])
def test_few_border_unknowns(buses, shared):
    """Three cliques, the later ones joined to the first by `shared` of its buses: fronts
    with 2 to 8 border unknowns below a root."""
    rng = np.random.default_rng(buses + shared)
    core = list(range(buses))
    br, nb = fronts._clique(core, rng), buses
    for k in range(2):
        own = core[1 + k * shared:1 + (k + 1) * shared]
        new = list(range(nb, nb + buses - shared))
        nb += len(new)
        br += [e for e in fronts._clique(own + new, rng) if not (e[0] in own and e[1] in own)]
    bt = np.ones(nb, np.int32)
    bt[0] = 3
    fronts._check(make_grid(nb, br), bt)
