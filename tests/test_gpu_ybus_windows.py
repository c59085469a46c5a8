"""The Ybus method on windows (ybus_fused = 1: row sums of V_i conj(Y_ij V_j))
against its separate form (ybus_fused = 0: row currents from the CSR row
kernels) over the states and grids that leave its usual path: parallel runs, a
hub window, isolated buses, zero and extreme magnitudes, non-finite angles.
"""
import numpy as np
import pytest

from gridcases import hub_grid, make_grid, random_grid, random_state, three_bus_plus

pytestmark = pytest.mark.gpu

# Every product is within 2^-52 of its magnitude and a row of n entries adds n
# of them, two or three roundings each: n 2^-50 of the row's largest term bounds
# both forms' error, and the hub's row has 441 entries.
TOL = 2.0 * 441 * 2.0**-50


@pytest.fixture(scope="module")
def pf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2302_10736_gb300 import pfgrid
    return pfgrid


def _states(nb, seed):
    vm, va = random_state(nb, seed)
    yield "usual", vm, va
    rng = np.random.default_rng(seed)
    for name, val in (("zero", 0.0), ("subnormal", 1e-310), ("tiny", 1e-200), ("below_mid", 2.0**-301),
                      ("huge", 1e120), ("above_mid", 2.0**301), ("negative", -1.02), ("nan_v", np.nan)):
        v = vm.copy()
        v[rng.choice(nb, max(1, nb // 10), replace=False)] = val
        yield name, v, va
    for name, val in (("far_angle", 1e7), ("nan_angle", np.nan), ("inf_angle", np.inf)):
        a = va.copy()
        a[rng.choice(nb, max(1, nb // 10), replace=False)] = val
        yield name, vm, a


def _grid(which):
    if which == "hub":
        return hub_grid(400, 3)
    if which == "parallel":
        return three_bus_plus()
    if which == "no_branches":
        return make_grid(3, [], shunts={0: (0.1, 0.2), 2: (0.0, -0.3)})
    gr = random_grid(700, 930, 11, shift_max=0.2)
    if which == "constants":   # branch constants at and beyond the fixed-point range
        gr["g"][::17], gr["b"][::17] = 1e-295, -1e-300
        gr["g"][5::17], gr["b"][5::17] = 3e90, -1e95
    return gr


@pytest.mark.parametrize("which", ["random", "constants", "hub", "parallel", "no_branches"])
@pytest.mark.parametrize("window", [128, 256])
def test_windows_equal_the_row_kernels(pf, which, window):
    import torch
    gr = _grid(which)
    nb = gr["nb"]
    grid = pf.ybus_build(gr)
    pf.grid_set_config(grid, ew_window=window, ybus_lanes=1, ybus_block=128)
    rp = pf.ybus_get(grid)[0].cpu().numpy()
    row = np.repeat(np.arange(nb), np.diff(rp))
    e = np.arange(len(row))
    at = [rp[row] + e, rp[row] + e + np.diff(rp)[row]]   # the theta and the v entries of the two halves
    dev = lambda x: torch.tensor(x, dtype=torch.float64, device="cuda")
    for name, vm, va in _states(nb, 5):
        got = []
        for fused in (0, 1):
            pf.grid_set_config(grid, ybus_fused=fused)
            P, Q, J = (torch.full((n,), 7.0, dtype=torch.float64, device="cuda") for n in (nb, nb, grid.nnzJ))
            Pi, Qi = torch.full_like(P, 7.0), torch.full_like(P, 7.0)
            pf.jac_ybus(grid, dev(vm), dev(va), P, Q, J)
            pf.inj_ybus(grid, dev(vm), dev(va), Pi, Qi)
            got.append([x.cpu().numpy() for x in (P, Q, J, Pi, Qi)])
        ref, new = got
        for x, y in zip(new, ref):
            assert np.array_equal(np.isnan(x), np.isnan(y)), name
        with np.errstate(invalid="ignore", over="ignore"):
            halves = [r.reshape(2, -1)[:, a] for r in (ref[2], new[2]) for a in at]   # [theta, v] of ref, then of new
            scale = []
            for k in (0, 1):
                m = np.zeros(nb)
                np.maximum.at(m, row, np.nan_to_num(np.abs(halves[k]).max(axis=0), posinf=np.inf))
                scale.append(m)
            # the separate form's diagonal j (S_i - v_i V_i conj(Y_ii U_i)) takes v_i^2 Y_ii in and out again: v_i
            # times the row's dS/dv belongs to the terms of its theta entries
            scale[0] += np.abs(np.nan_to_num(vm)) * np.nan_to_num(scale[1], posinf=0.0)
            for k in (0, 1):
                d = np.abs(halves[2 + k] - halves[k])
                assert np.nanmax(np.where(np.isfinite(d), d - TOL * scale[k][row], -1.0)) <= 0.0, (name, k)
            # S_i is the sum of the row's v_j dS_i/dv_j: its terms are the theta entries and v_i times the diagonal's
            big = scale[0] + np.abs(np.nan_to_num(ref[0])) + np.abs(np.nan_to_num(ref[1]))
            for k in (0, 1, 3, 4):
                d = np.abs(new[k] - ref[k % 3])
                assert np.nanmax(np.where(np.isfinite(d), d - TOL * big, -1.0)) <= 0.0, (name, k)
    pf.grid_check_error(grid)
