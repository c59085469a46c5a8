"""Runs of parallel branches in the element-wise Jacobians (GPU).

The first branch's thread adds its run's later branches onto the entries, and
the bus sums run along the staged rows, where an outage inside a run leaves the
entry with the others.  Against the oracle at the repository's 1e-12, with runs
of 2 to 6 branches in both orientations over every cut into windows; a scenario
without an outage equals the single evaluation bit for bit.
"""
import numpy as np
import pytest

from gridcases import random_grid, random_state
from test_gpu_batched import _d, check_batch, pf  # noqa: F401  (pf: fixture)
from test_gpu_parity import check_against_oracle

pytestmark = pytest.mark.gpu


def with_runs(gr, seed, share):
    """A share of the branches repeated 1 to 5 times, some of them reversed."""
    rng = np.random.default_rng(seed)
    pick = np.flatnonzero(rng.random(gr["nl"]) < share)
    src = np.repeat(pick, rng.integers(1, 6, pick.size))
    out = dict(gr)
    for k in ("f", "t", "g", "b", "bsh", "tap", "shift"):
        v = gr[k][src]
        if k in ("g", "b"):
            v = v * rng.uniform(0.5, 1.5, src.size)
        out[k] = np.concatenate([gr[k], v]).astype(gr[k].dtype)
    rev = gr["nl"] + np.flatnonzero(rng.random(src.size) < 0.5)
    out["f"][rev], out["t"][rev] = out["t"][rev].copy(), out["f"][rev].copy()
    out["nl"] = gr["nl"] + src.size
    return out, src


@pytest.mark.parametrize("nb,nl,share,window", [(5, 6, 1.0, 128), (130, 180, 0.9, 128), (130, 180, 0.9, 256),
                                                (3000, 4000, 0.3, 256)])
def test_runs(pf, nb, nl, share, window):  # noqa: F811
    import torch
    gr, src = with_runs(random_grid(nb, nl, 7, shift_max=0.2), nb, share)
    vm, va = random_state(nb, 3)
    grid = pf.ybus_build(gr)
    pf.grid_set_config(grid, ew_window=window)
    check_against_oracle(pf, gr, vm, va, grid=grid)
    # out: none, the first, a middle and the last branch of a run, a single branch
    run = np.concatenate([[src[0]], nl + np.flatnonzero(src == src[0])])
    single = np.setdiff1d(np.arange(nl), src)
    out = [-1, run[0], run[len(run) // 2], run[-1]] + ([int(single[0])] if single.size else [])
    S = len(out)
    vms = np.stack([random_state(nb, 10 + s)[0] for s in range(S)])
    vas = np.stack([random_state(nb, 10 + s)[1] for s in range(S)])
    check_batch(pf, gr, vms, vas, np.array(out, np.int32))
    P1, Q1 = (torch.empty(nb, dtype=torch.float64, device="cuda") for _ in range(2))
    J1 = torch.empty(grid.nnzJ, dtype=torch.float64, device="cuda")
    for tb, tf in ((128, 1), (128, 3), (256, 2)):
        batch = pf.batch_create(grid, S, np.array(out, np.int32))
        pf.batch_set_config(batch, window=tb, terminals_per_thread=tf)
        P, Q = (torch.empty(S * nb, dtype=torch.float64, device="cuda") for _ in range(2))
        J = torch.empty(batch.nnzJ_total, dtype=torch.float64, device="cuda")
        pf.jac_elementwise_batched(batch, _d(vms.reshape(-1)), _d(vas.reshape(-1)), P, Q, J)
        pf.jac_elementwise(grid, _d(vms[0]), _d(vas[0]), P1, Q1, J1)
        torch.cuda.synchronize()
        assert torch.equal(P[:nb], P1) and torch.equal(Q[:nb], Q1) and torch.equal(J[:grid.nnzJ], J1), (tb, tf)
