"""The Ybus method with branches out of service (zero constants) and dead buses
(zero magnitude): against the separate form, and on the usual path.
"""
import numpy as np
import pytest

from gridcases import random_grid, random_state
from test_gpu_parallel_runs import with_runs
from test_gpu_ybus_windows import TOL

pytestmark = pytest.mark.gpu


def _dev(x):
    import torch
    return torch.tensor(x, dtype=torch.float64, device="cuda")


def _out_of_service(gr, share, seed):
    off = np.random.default_rng(seed).random(gr["nl"]) < share
    return dict(gr, **{k: np.where(off, 0.0, gr[k]) for k in ("g", "b", "bsh")})


@pytest.mark.parametrize("nb,nl", [(40, 56), (3000, 4000)])
@pytest.mark.parametrize("share", [0.02, 0.4, 1.0])
@pytest.mark.parametrize("dead", [0.0, 0.1, 1.0])
def test_zero_entries_and_magnitudes(nb, nl, share, dead):
    """Runs of parallel branches, whole or in part out of service, beside live and
    dead buses; bounds of test_gpu_ybus_windows (every entry against its row's
    largest term)."""
    import torch
    from paper_2302_10736_gb300 import pfgrid as pf
    gr = _out_of_service(with_runs(random_grid(nb, nl, 7, shift_max=0.2), nb, 0.3)[0], share, nl)
    vm, va = random_state(nb, 3)
    vm = np.where(np.random.default_rng(nb).random(nb) < dead, 0.0, vm)
    grid = pf.ybus_build(gr)
    rp = pf.ybus_get(grid)[0].cpu().numpy()
    row = np.repeat(np.arange(nb), np.diff(rp))
    e = np.arange(len(row))
    at = [rp[row] + e, rp[row] + e + np.diff(rp)[row]]
    got = []
    for fused in (0, 1):
        pf.grid_set_config(grid, ybus_fused=fused, ybus_lanes=1, ybus_block=128)
        P, Q, J = (torch.full((n,), 7.0, dtype=torch.float64, device="cuda") for n in (nb, nb, grid.nnzJ))
        Pi, Qi = torch.full_like(P, 7.0), torch.full_like(P, 7.0)
        pf.jac_ybus(grid, _dev(vm), _dev(va), P, Q, J)
        pf.inj_ybus(grid, _dev(vm), _dev(va), Pi, Qi)
        got.append([x.cpu().numpy() for x in (P, Q, J, Pi, Qi)])
    ref, new = got
    halves = [r.reshape(2, -1)[:, a] for r in (ref[2], new[2]) for a in at]
    scale = []
    for k in (0, 1):
        m = np.zeros(nb)
        np.maximum.at(m, row, np.abs(halves[k]).max(axis=0))
        scale.append(m)
    scale[0] = scale[0] + np.abs(vm) * scale[1]
    for k in (0, 1):
        assert (np.abs(halves[2 + k] - halves[k]) <= TOL * scale[k][row][None]).all(), k
    big = scale[0] + np.abs(ref[0]) + np.abs(ref[1])
    for k in (0, 1, 3, 4):
        assert (np.abs(new[k] - ref[k % 3]) <= TOL * big).all(), k


def test_branches_out_of_service_stay_on_the_usual_path():
    """1 % of the branches out of service do not change the time of an evaluation
    (as rows evaluated whole they made it four times as long)."""
    import torch
    from paper_2302_10736_gb300 import pfgrid as pf
    nb, nl = 70000, 88000
    gr = random_grid(nb, nl, 9)
    at = tuple(_dev(x) for x in random_state(nb, 3))
    ms = []
    for g in (gr, _out_of_service(gr, 0.01, 1)):
        grid = pf.ybus_build(g)
        P, Q, J = (torch.empty(n, dtype=torch.float64, device="cuda") for n in (nb, nb, grid.nnzJ))
        best = []
        for _ in range(5):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            pf.jac_ybus(grid, *at, P, Q, J)
            e0.record()
            for _ in range(100):
                pf.jac_ybus(grid, *at, P, Q, J)
            e1.record()
            torch.cuda.synchronize()
            best.append(e0.elapsed_time(e1))
        ms.append(min(best))
    assert ms[1] <= 1.5 * ms[0]
