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
    """grid_autotune settles the windows before it times the Ybus form that runs on
    them (one launch; the other form's row kernel comes after a phasor launch)."""
    from paper_2302_10736_gb300 import pfgrid as pf
    grid = pf.ybus_build(random_grid(700, 930, 9))
    vm, va = (_dev(x) for x in random_state(700, 1))
    pf.grid_trace_enable(grid, 1 << 14)
    best = pf.grid_autotune(grid, vm, va, reps=2)
    names = [k for k, _ in pf.grid_trace_read(grid)]
    assert "jac_ew" in names and "jac_ybus" in names
    one = [i for i, k in enumerate(names) if k == "jac_ybus" and (i == 0 or names[i - 1] != "phasor")]
    assert one and max(i for i, k in enumerate(names) if k == "jac_ew") < one[0]
    assert pf.grid_get_config(grid) == best
    assert max(pf.grid_ew_windows(grid)[:, 3]) <= best["ew_window"]   # the layout in place is the one named


def test_shape_a_batch_starts_from():
    """By size unless the program has set another shape than the initial one,
    however it came to the present one."""
    from paper_2302_10736_gb300 import pfgrid as pf
    nb = 700
    grid = pf.ybus_build(random_grid(nb, 930, 9))

    def shape():
        c = pf.batch_get_config(pf.batch_create(grid, 3))
        return c["ybus_lanes"], c["ybus_block"]

    by_size = shape()
    assert by_size[1] == 64
    first = pf.grid_get_config(grid)
    pf.grid_set_config(grid, **first)   # the initial shape, named
    assert shape() == by_size
    pf.grid_set_config(grid, ybus_lanes=16, ybus_block=128)
    assert shape() == (16, 128)
    pf.grid_set_config(grid, ew_window=128)   # something else
    assert shape() == (16, 128)
    pf.grid_set_config(grid, **first)   # and back
    assert shape() == by_size
    pf.grid_set_config(grid, ybus_lanes=16, ybus_block=128)
    pf.grid_autotune(grid, *(_dev(x) for x in random_state(nb, 1)), reps=1)   # one state's shape
    assert shape() == by_size
    pf.grid_set_config(grid, ew_window=128)
    assert shape() == by_size
    lanes = 32 if pf.grid_get_config(grid)["ybus_lanes"] != 32 else 16   # another than the tuner's
    pf.grid_set_config(grid, ybus_lanes=lanes, ybus_block=512)
    assert shape() == (lanes, 512)


def test_batch_tuner_times_the_present_shape_and_64_threads():
    """batch_autotune's Ybus candidates: the shape in place, and 6 lane counts by 4
    CTA sizes, the default one (64 threads) among them; each is launched once and
    then timed."""
    from paper_2302_10736_gb300 import pfgrid as pf
    nb, S, reps = 300, 4, 3
    grid = pf.ybus_build(random_grid(nb, 420, 9))
    batch = pf.batch_create(grid, S)
    pf.batch_set_config(batch, ybus_lanes=2, ybus_block=96)
    vm, va = random_state(nb, 1, S)
    pf.grid_trace_enable(grid, 1 << 12)
    pf.batch_autotune(batch, _dev(vm.ravel()), _dev(va.ravel()), reps=reps, kernels=2)
    names = [k for k, _ in pf.grid_trace_read(grid)]
    assert names == ["jac_ybus_batched"] * ((1 + 6 * 4) * (1 + reps))
