"""Calls issued back to back on one stream, each kernel launched as a
programmatic dependent of the one before: every call sees its own state, not
what an earlier call left in the shared phasor workspace.
"""
import numpy as np
import pytest

from gridcases import random_grid, random_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb,nl", [(700, 930), (40, 55), (5000, 6600)])
@pytest.mark.parametrize("jac", [True, False])
def test_ybus_rows_back_to_back(nb, nl, jac):
    """Alternating states through one batch and through one grid's separate
    form: results equal those of the first, waited-for call bit for bit."""
    import torch
    from paper_2302_10736_gb300 import pfgrid as pf
    grid = pf.ybus_build(random_grid(nb, nl, 9))
    pf.grid_set_config(grid, ybus_fused=0)
    batch = pf.batch_create(grid, 1)
    dev = lambda x: torch.tensor(x, dtype=torch.float64, device="cuda")
    new = lambda n: torch.full((n,), 7.0, dtype=torch.float64, device="cuda")
    states = [tuple(dev(x) for x in random_state(nb, seed)) for seed in (1, 2)]

    def call(on, st, out):
        fn = {(True, True): pf.jac_ybus_batched, (True, False): pf.inj_ybus_batched,
              (False, True): pf.jac_ybus, (False, False): pf.inj_ybus}[on is batch, jac]
        fn(on, *st, *out)

    for on in (batch, grid):
        size = (nb, nb, grid.nnzJ) if jac else (nb, nb)
        ref = [[new(n) for n in size] for _ in states]
        for st, out in zip(states, ref):
            call(on, st, out)
            torch.cuda.synchronize()
        outs = [[new(n) for n in size] for _ in range(200)]
        for k, out in enumerate(outs):
            call(on, states[k % 2], out)
        torch.cuda.synchronize()
        for k, out in enumerate(outs):
            for x, y in zip(out, ref[k % 2]):
                assert torch.equal(x, y), (k, int((x != y).sum()))


def test_reduced_system_back_to_back():
    """The same for the Ybus method's reduced system (evaluation, then gather)."""
    import torch
    from paper_2302_10736_gb300 import pfgrid as pf
    nb = 5000
    gr = random_grid(nb, 6600, 9)
    dev = lambda x: torch.tensor(x, dtype=torch.float64, device="cuda")
    new = lambda n: torch.full((n,), 7.0, dtype=torch.float64, device="cuda")
    states = [tuple(dev(x) for x in random_state(nb, seed)) for seed in (1, 2)]
    spec = [dev(np.full(nb, 0.5)), dev(np.full(nb, -0.25))]
    for fused in (0, 1):
        grid = pf.ybus_build(gr)
        pf.grid_set_config(grid, ybus_fused=fused)
        pf.grid_set_bus_types(grid, gr["bustype"])
        n, _, nnz = pf.jac_reduced_info(grid)
        ref = [(new(n), new(nnz)) for _ in states]
        for st, out in zip(states, ref):
            pf.jac_reduced(grid, "ybus", *st, *spec, *out)
            torch.cuda.synchronize()
        outs = [(new(n), new(nnz)) for _ in range(200)]
        for k, out in enumerate(outs):
            pf.jac_reduced(grid, "ybus", *states[k % 2], *spec, *out)
        torch.cuda.synchronize()
        for k, out in enumerate(outs):
            for x, y in zip(out, ref[k % 2]):
                assert torch.equal(x, y), (fused, k, int((x != y).sum()))
