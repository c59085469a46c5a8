"""jac_reduced_solve on grids whose fronts lie at the edges of the kernels that
eliminate them: a complete graph is one front of all its unknowns.  Against
LAPACK's pivoting dense solve; tolerances as in test_gpu_reduced (solution 1e-10
of its largest entry, normwise backward error 1e-13), two solves bitwise equal.
"""
import numpy as np
import pytest

from gridcases import make_grid, series

pytestmark = pytest.mark.gpu


def _clique(buses, rng, scale=1.0):
    br = []
    for x, i in enumerate(buses):
        for j in buses[x + 1:]:
            g, b = series(rng.uniform(0.001, 0.05), rng.uniform(0.01, 0.3))
            br.append((i, j, scale * g, scale * b, rng.uniform(0, 0.1), 1.0, 0.0))
    return br


def _check(gr, bt):
    import torch
    import scipy.sparse as sp
    from paper_2302_10736_gb300 import pfgrid as pf
    nb = gr["nb"]
    rng = np.random.default_rng(nb)
    dev = lambda x: torch.tensor(x, dtype=torch.float64, device="cuda")
    grid = pf.ybus_build(gr)
    pf.grid_set_bus_types(grid, bt)
    n, _, nnz = pf.jac_reduced_info(grid)
    F, dx, dx2 = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(3))
    Jr = torch.empty(nnz, dtype=torch.float64, device="cuda")
    vm, va = dev(rng.uniform(0.97, 1.03, nb)), dev(rng.normal(0, 0.02, nb))
    pf.jac_reduced(grid, "elementwise", vm, va, dev(rng.normal(size=nb)), dev(rng.normal(size=nb)), F, Jr)
    for out in (dx, dx2):
        pf.jac_reduced_solve(grid, Jr, F, out)
    pf.grid_check_error(grid)
    assert torch.equal(dx, dx2)
    cp, ri = pf.jac_reduced_pattern(grid)
    A = sp.csc_matrix((Jr.cpu().numpy(), ri, cp), shape=(n, n)).toarray()
    x, Fh = dx.cpu().numpy(), F.cpu().numpy()
    ref = np.linalg.solve(A, Fh)
    assert np.max(np.abs(x - ref)) <= 1e-10 * np.max(np.abs(ref))
    back = np.max(np.abs(A @ x - Fh)) / (np.max(np.abs(A).sum(axis=1)) * np.max(np.abs(x)) + np.max(np.abs(Fh)))
    assert back <= 1e-13
    return n


@pytest.mark.parametrize("n", [1, 2, 12, 13, 31, 32, 63, 64, 127, 128, 191, 192, 255, 256])
def test_one_front(n):
    """A complete graph with n unknowns."""
    nb = n // 2 + n % 2 + 1
    bt = np.ones(nb, np.int32)
    bt[0] = 3
    if n % 2:
        bt[1] = 2   # a PV bus has an angle only
    rng = np.random.default_rng(n)
    assert _check(make_grid(nb, _clique(list(range(nb)), rng)), bt) == n


@pytest.mark.parametrize("core,arm", [(6, 5), (14, 20), (30, 14), (62, 33), (70, 60), (126, 40)])
def test_fronts_below_a_front(core, arm):
    """Cliques of `arm` buses hung on parts of a clique of `core` buses (their
    updates reach the core's front from fronts of another class), some of them
    on the same buses, and radial buses on those."""
    rng = np.random.default_rng(core)
    br = _clique(list(range(core)), rng)
    nb = core
    for k in range(4):
        at = sorted(rng.choice(core, max(2, core // (3 if k else 2)), replace=False).tolist()) if k != 3 else at
        new = list(range(nb, nb + arm))
        nb += arm
        br += _clique(new, rng) + [(at[i % len(at)], new[i % arm]) + series(0.01, 0.1) + (0.02, 1.0, 0.0)
                                   for i in range(max(len(at), arm))]
        for i in new[::3]:
            br.append((i, nb) + series(0.02, 0.15) + (0.01, 1.0, 0.0))
            nb += 1
    bt = np.ones(nb, np.int32)
    bt[0] = 3
    bt[2::5] = 2
    _check(make_grid(nb, br), bt)
