"""Calls issued back to back whose inputs the call just before writes (targets,
parameters): as when each is waited for.  The kernels are launched as programmatic
dependents of one another, and may start before that call is done.
"""
import numpy as np
import pytest

from gridcases import random_grid, random_state

pytestmark = pytest.mark.gpu

NB, NL, N = 5000, 6600, 100


def _dev(x):
    import torch
    return torch.tensor(x, dtype=torch.float64, device="cuda")


def _new(n):
    import torch
    return torch.full((n,), 7.0, dtype=torch.float64, device="cuda")


def _equal_runs(calls, sizes):
    """calls(k, out) issues pass k; back to back as waited for."""
    import torch
    ref = [[_new(n) for n in sizes] for _ in range(2)]
    for k, out in enumerate(ref):
        calls(k, out)
        torch.cuda.synchronize()
    outs = [[_new(n) for n in sizes] for _ in range(N)]
    for k, out in enumerate(outs):
        calls(k % 2, out)
    torch.cuda.synchronize()
    for k, out in enumerate(outs):
        for x, y in zip(out, ref[k % 2]):
            assert torch.equal(x, y), (k, int((x != y).sum()))


@pytest.mark.parametrize("method", ["ybus", "elementwise"])
@pytest.mark.parametrize("fused", [0, 1])
def test_targets_written_just_before(method, fused):
    from paper_2302_10736_gb300 import pfgrid as pf
    gr = random_grid(NB, NL, 9)
    grid = pf.ybus_build(gr)
    pf.grid_set_config(grid, ybus_fused=fused)
    pf.grid_set_bus_types(grid, gr["bustype"])
    n, _, nnz = pf.jac_reduced_info(grid)
    goal = [tuple(_dev(x) for x in random_state(NB, s)) for s in (1, 2)]
    at = tuple(_dev(x) for x in random_state(NB, 3))
    Ps, Qs = _new(NB), _new(NB)
    inj = pf.inj_ybus if method == "ybus" else pf.inj_elementwise

    def calls(k, out):
        inj(grid, *goal[k], Ps, Qs)
        pf.jac_reduced(grid, method, *at, Ps, Qs, *out)

    _equal_runs(calls, (n, nnz))


@pytest.mark.parametrize("jac", [True, False])
@pytest.mark.parametrize("what", ["batch", "rows", "windows", "elementwise"])
def test_parameters_set_just_before(what, jac):
    from paper_2302_10736_gb300 import pfgrid as pf
    gr = random_grid(NB, NL, 9, shift_max=0.2)
    grid = pf.ybus_build(gr)
    pf.grid_set_config(grid, ybus_fused=int(what == "windows"))
    on = pf.batch_create(grid, 1, np.array([17], np.int32)) if what == "batch" else grid
    params = [[_dev(gr[k] * f) for k in ("g", "b", "bsh", "tap", "shift", "gs", "bs")] for f in (1.0, 1.01)]
    at = tuple(_dev(x) for x in random_state(NB, 3))
    fn = {("batch", True): pf.jac_ybus_batched, ("batch", False): pf.inj_ybus_batched,
          ("elementwise", True): pf.jac_elementwise, ("elementwise", False): pf.inj_elementwise}.get(
              (what, jac), pf.jac_ybus if jac else pf.inj_ybus)

    def calls(k, out):
        pf.grid_set_params(grid, *params[k])
        fn(on, *at, *out)

    _equal_runs(calls, (NB, NB, on.nnzJ_total if what == "batch" else grid.nnzJ) if jac else (NB, NB))
