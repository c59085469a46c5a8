"""jac_reduced_solve on fronts far beyond what a cluster of CTAs holds: complete
graphs, one front of all their unknowns.  Checks and tolerances of
test_gpu_lu_fronts.
"""
import pytest

import test_gpu_lu_fronts as fronts

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1201, 1202])
def test_one_front_above_1200_unknowns(n):
    """Every pivot block, not only those that fit shared memory."""
    fronts.test_one_front(n)
