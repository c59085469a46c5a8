"""The Ybus method on windows against its separate form where results leave the
doubles' range: the same entries overflow, to the same infinity, and the same
ones are not a number.  States and grids of test_gpu_ybus_windows, and infinite
and near-overflowing magnitudes besides.
"""
import numpy as np
import pytest

from gridcases import random_state
from test_gpu_ybus_windows import TOL, _grid, _states, pf  # noqa: F401  (pf: fixture)

pytestmark = pytest.mark.gpu


def _more_states(nb, seed):
    vm, va = random_state(nb, seed)
    rng = np.random.default_rng(seed + 1)
    for name, val in (("inf_v", np.inf), ("minus_inf_v", -np.inf), ("above_square", 1e170), ("near_largest", 1e300)):
        v = vm.copy()
        v[rng.choice(nb, max(1, nb // 10), replace=False)] = val
        yield name, v, va


@pytest.mark.parametrize("which", ["random", "constants", "hub", "parallel", "no_branches"])
@pytest.mark.parametrize("window", [128, 256])
def test_same_infinities(pf, which, window):  # noqa: F811
    import torch
    gr = _grid(which)
    nb = gr["nb"]
    grid = pf.ybus_build(gr)
    pf.grid_set_config(grid, ew_window=window, ybus_lanes=1, ybus_block=128)
    rp = pf.ybus_get(grid)[0].cpu().numpy()
    row = np.repeat(np.arange(nb), np.diff(rp))
    e = np.arange(len(row))
    at = [rp[row] + e, rp[row] + e + np.diff(rp)[row]]
    dev = lambda x: torch.tensor(x, dtype=torch.float64, device="cuda")
    for name, vm, va in list(_states(nb, 5)) + list(_more_states(nb, 5)):
        got = []
        for fused in (0, 1):
            pf.grid_set_config(grid, ybus_fused=fused)
            P, Q, J = (torch.full((n,), 7.0, dtype=torch.float64, device="cuda") for n in (nb, nb, grid.nnzJ))
            Pi, Qi = torch.full_like(P, 7.0), torch.full_like(P, 7.0)
            pf.jac_ybus(grid, dev(vm), dev(va), P, Q, J)
            pf.inj_ybus(grid, dev(vm), dev(va), Pi, Qi)
            got.append([x.cpu().numpy() for x in (P, Q, J, Pi, Qi)])
        ref, new = got
        for k, (x, y) in enumerate(zip(new, ref)):
            assert np.array_equal(np.isnan(x), np.isnan(y)), (name, k)
            assert np.array_equal(np.isinf(x), np.isinf(y)), (name, k)
            assert np.array_equal(x[np.isinf(x)], y[np.isinf(y)]), (name, k)
        # finite entries against the row's largest finite term, each half and kind
        # of entry apart (as in test_gpu_ybus_windows, theta's with v_i times v's)
        halves = [r.reshape(2, -1)[:, a] for r in (ref[2], new[2]) for a in at]
        scale = []
        for k in (0, 1):
            m = np.zeros(nb)
            fin = np.where(np.isfinite(halves[k]), np.abs(halves[k]), 0.0).max(axis=0)
            np.maximum.at(m, row, fin)
            scale.append(m)
        with np.errstate(over="ignore"):
            scale[0] = scale[0] + np.where(np.isfinite(vm), np.abs(vm), 0.0) * scale[1]
        for k in (0, 1):
            ok = np.isfinite(halves[k]) & np.isfinite(scale[k][row])[None]
            d = np.abs(np.where(ok, halves[2 + k], 0.0) - np.where(ok, halves[k], 0.0))
            assert (d <= np.where(ok, TOL * scale[k][row][None], 0.0)).all(), (name, k)
    pf.grid_check_error(grid)
