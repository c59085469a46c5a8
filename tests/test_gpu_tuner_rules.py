"""What the launch-shape tuners time, in which order, and which shape a batch's
Ybus row kernels start from.
"""
import pytest

from gridcases import random_grid, random_state

pytestmark = pytest.mark.gpu


def _dev(x):
    import torch
    return torch.tensor(x, dtype=torch.float64, device="cuda")


def test_ybus_form_is_timed_on_the_windows_kept():
    """grid_autotune settles the windows before it times the Ybus forms, one of
    which runs on them."""
    from paper_2302_10736_gb300 import pfgrid as pf
    grid = pf.ybus_build(random_grid(700, 930, 9))
    vm, va = (_dev(x) for x in random_state(700, 1))
    pf.grid_trace_enable(grid, 1 << 14)
    best = pf.grid_autotune(grid, vm, va, reps=2)
    names = [k for k, _ in pf.grid_trace_read(grid)]
    assert "jac_ew" in names and "jac_ybus" in names
    assert max(i for i, k in enumerate(names) if k == "jac_ew") < names.index("jac_ybus")
    assert pf.grid_get_config(grid) == best
    assert max(pf.grid_ew_windows(grid)[:, 3]) <= best["ew_window"]   # the layout in place is the one named
