"""The work that is timed: what programs have this library do, through its public entry points.

Every case is a grid (nb buses, nl branches, drawn by the repository's seeded generator), voltage states and one of
the calls of `KINDS`.  Sizes are those of the tests and of bench.py: the paper's bus counts with 1.32 branches per
bus, and the numbered workloads of paper_2302_10736_gb300/synth.  All values are FP64 (the library has no other
type).  A grid, its states and the handles a program keeps (grid, batch, bus types) are made in prepare(); run() is
one call, or the few calls of one step.
"""
import numpy as np
import torch

from paper_2302_10736_gb300 import pfgrid, synth

KINDS = {
    "jac": "bus injections and Jacobian values of one state, element-wise method (jac_elementwise)",
    "inj": "bus injections of one state, element-wise method (inj_elementwise)",
    "ybus_jac": "bus injections and Jacobian values of one state, Ybus method (jac_ybus)",
    "ybus_inj": "bus injections of one state, Ybus method (inj_ybus)",
    "host": "injections and Jacobian values from and to page-locked host buffers, waited for (eval_host)",
    "n1": "injections and Jacobians of nscen N-1 contingencies, element-wise method (jac_elementwise_batched)",
    "n1_ybus": "the same by the Ybus method (jac_ybus_batched)",
    "loss_grad": "a training step: mismatch loss and all its gradients through autograd (MismatchLoss)",
    "adjoint": "losses and gradients of nscen states on one grid (adjoint_elementwise)",
    "newton_step": "one Newton step: mismatch, reduced Jacobian and the solve (jac_reduced, jac_reduced_solve)",
    "powerflow": "a Newton power flow to max |F| <= 1e-10 (powerflow_newton)",
}


def listed():
    def case(name, kind, nb, nl, nscen=1, shift=0.0, random_order=False, pv=0.2):
        return dict(name=name, kind=kind, nb=nb, nl=nl, nscen=nscen, shift=shift, random_order=random_order, pv=pv)

    return [
        # the smallest calls: a study that evaluates a teaching-size network over and over; latency only
        case("jac-118", "jac", 118, 156),
        # the headline: one state of a continental grid, everything a Newton or sensitivity program reads
        case("jac-70k", "jac", 70000, 88000, pv=0.15),
        # mismatch checks of a mid-size grid with phase shifters: injections without a Jacobian
        case("inj-9241", "inj", 9241, 12198, shift=0.2),
        # the same two by the Ybus method, which programs with an admittance matrix in hand use
        case("ybus-jac-70k", "ybus_jac", 70000, 88000, pv=0.15),
        case("ybus-inj-25k", "ybus_inj", 25000, 33000),
        # a CPU program that calls the library once per iteration: inputs and results in its own page-locked memory
        case("host-70k", "host", 70000, 88000, pv=0.15),
        # contingency screening: every state with a branch of its own out
        case("n1-10k-x1024", "n1", 10000, 13500, nscen=1024),
        case("n1-ybus-10k-x256", "n1_ybus", 10000, 13500, nscen=256),
        # learning states and branch parameters: one forward and backward pass of the loss
        case("loss-grad-25k", "loss_grad", 25000, 33000),
        # state estimation over many snapshots of a very large grid (the largest working set per state)
        case("adjoint-250k-x16", "adjoint", 250000, 330000, nscen=16),
        # one step of a caller's own Newton loop, and a whole power flow
        case("newton-step-25k", "newton_step", 25000, 33000),
        case("powerflow-10k", "powerflow", 10000, 13500),
    ]


# per kind: the range of buses, and of states times buses (a drawn case costs no more than the largest listed one)
RANGES = {
    "jac": (14, 410000), "inj": (14, 410000), "ybus_jac": (14, 410000), "ybus_inj": (14, 410000),
    "host": (118, 164000), "n1": (118, 25000), "n1_ybus": (118, 25000), "loss_grad": (118, 82000),
    "adjoint": (300, 250000), "newton_step": (118, 25000), "powerflow": (118, 10000),
}


def draw(rng):
    kind = rng.choice(sorted(KINDS))
    lo, hi = RANGES[kind]
    nb = int(round(lo * (hi / lo) ** rng.random()))
    nl = max(nb + 4, int(round(nb * rng.uniform(1.2, 1.4))))
    nscen = 1
    if kind in ("n1", "n1_ybus", "adjoint"):
        most = min({"n1": 2048, "n1_ybus": 1024, "adjoint": 64}[kind], (4000000 if kind == "adjoint" else 8000000) // nb)
        if kind != "adjoint":
            most = min(most, max(1, nl - nb) // 2)   # distinct branches that are no bridges
        nscen = int(round(most ** rng.random()))
    return dict(kind=kind, nb=nb, nl=nl, nscen=max(1, nscen), shift=rng.choice([0.0, 0.2]),
                random_order=rng.random() < 0.25, pv=round(rng.uniform(0.1, 0.25), 3))


def _inputs(case, seed):
    """The grid and states of a case as host arrays, from the seed alone."""
    kind, nb, nl, S = case["kind"], case["nb"], case["nl"], case["nscen"]
    seed = synth.BASE_SEED + 1000 * int(seed)
    # the Newton cases solve one network for many states (the length of their results depends on its bus types)
    net = synth.BASE_SEED if kind in ("newton_step", "powerflow") else seed
    gr = synth.grid(nb, nl, net, shift_max=case["shift"], pv_frac=case["pv"])
    if kind in ("n1", "n1_ybus"):
        gr["vm"], gr["va"] = synth.voltages(nb, S, seed, 0, 0.93, 1.07, 0.25)
        gr["outage"] = synth.outages(synth.bridges(nb, gr["f"], gr["t"]), S, seed)
    else:
        gr["vm"], gr["va"] = synth.voltages(nb, S, seed)
    if kind in ("loss_grad", "adjoint"):
        vm2, va2 = synth.voltages(nb, 1, seed, 1)
        gr["vm2"], gr["va2"] = vm2[0], va2[0]
        gr["wP"], gr["wQ"] = synth.weights(nb, seed)
    if kind in ("newton_step", "powerflow"):
        # an operating point with moderate angles, and a start near it (the previous solution of a time series)
        rng = np.random.default_rng(seed)
        gr["vm2"], gr["va2"] = gr["vm"][0].copy(), 0.1 * gr["va"][0]
        bt = gr["bustype"]
        gr["vm"] = gr["vm2"] + np.where(bt == 1, rng.uniform(-1e-3, 1e-3, nb), 0.0)
        gr["va"] = gr["va2"] + np.where(bt <= 2, rng.uniform(-1e-3, 1e-3, nb), 0.0)
        gr["vm"], gr["va"] = gr["vm"][None], gr["va"][None]
    if case["random_order"]:
        gr = synth.renumber_buses(gr, net)
    return gr


DEV = "cuda"


def _dev(x):
    return torch.tensor(np.ascontiguousarray(x), device=DEV)


def _empty(n):
    return torch.empty(n, dtype=torch.float64, device=DEV)


def _pinned(n):
    return torch.empty(n, dtype=torch.float64, pin_memory=True)


PARAMS = ("g", "b", "bsh", "tap", "shift", "gs", "bs")


def prepare(case, seed):
    kind, nb, S = case["kind"], case["nb"], case["nscen"]
    gr = _inputs(case, seed)
    grid = pfgrid.ybus_build(gr)
    st = dict(kind=kind, grid=grid)
    if kind == "host":
        keep = [_pinned(n) for n in (nb, nb, nb, nb, grid.nnzJ)]   # page-locked for as long as the state lives
        keep[0].copy_(torch.from_numpy(gr["vm"][0]))
        keep[1].copy_(torch.from_numpy(gr["va"][0]))
        st.update(keep=keep, bufs=[t.numpy() for t in keep])
        return st
    st.update(vm=_dev(gr["vm"]).reshape(-1), va=_dev(gr["va"]).reshape(-1))
    if kind in ("jac", "ybus_jac", "inj", "ybus_inj"):
        st.update(P=_empty(nb), Q=_empty(nb))
        if kind in ("jac", "ybus_jac"):
            st["J"] = _empty(grid.nnzJ)
    elif kind in ("n1", "n1_ybus"):
        batch = pfgrid.batch_create(grid, S, gr["outage"])
        st.update(batch=batch, P=_empty(S * nb), Q=_empty(S * nb), J=_empty(batch.nnzJ_total))
    elif kind in ("loss_grad", "adjoint"):
        batch = pfgrid.batch_create(grid, S)
        Ps, Qs = _targets(gr)
        st.update(batch=batch, data=[Ps, Qs, _dev(gr["wP"]), _dev(gr["wQ"])])
        if kind == "loss_grad":
            st["leaves"] = [st["vm"].requires_grad_(), st["va"].requires_grad_()]
            st["leaves"] += [_dev(gr[k]).requires_grad_() for k in PARAMS[:4]]
            st["fixed"] = [_dev(gr[k]) for k in PARAMS[4:]]
        else:
            st["out"] = [_empty(S), _empty(S * nb), _empty(S * nb)] + [_empty(case["nl"]) for _ in range(4)]
    else:
        pfgrid.grid_set_bus_types(grid, gr["bustype"])
        st["spec"] = _targets(gr)
        n, _, nnz = pfgrid.jac_reduced_info(grid)
        if kind == "newton_step":
            st.update(F=_empty(n), Jr=_empty(nnz), dx=_empty(n))
            run(st)   # the first solve analyses the pattern, as in the first step of a caller's loop
        else:
            st.update(vm0=st["vm"].clone(), va0=st["va"].clone())
    return st


def run(st):
    kind, grid = st["kind"], st["grid"]
    if kind == "jac":
        pfgrid.jac_elementwise(grid, st["vm"], st["va"], st["P"], st["Q"], st["J"])
        return st["P"], st["Q"], st["J"]
    if kind == "inj":
        pfgrid.inj_elementwise(grid, st["vm"], st["va"], st["P"], st["Q"])
        return st["P"], st["Q"]
    if kind == "ybus_jac":
        pfgrid.jac_ybus(grid, st["vm"], st["va"], st["P"], st["Q"], st["J"])
        return st["P"], st["Q"], st["J"]
    if kind == "ybus_inj":
        pfgrid.inj_ybus(grid, st["vm"], st["va"], st["P"], st["Q"])
        return st["P"], st["Q"]
    if kind == "host":
        pfgrid.eval_host(grid, "elementwise", *st["bufs"])
        return tuple(st["bufs"][2:])
    if kind == "n1":
        pfgrid.jac_elementwise_batched(st["batch"], st["vm"], st["va"], st["P"], st["Q"], st["J"])
        return st["P"], st["Q"], st["J"]
    if kind == "n1_ybus":
        pfgrid.jac_ybus_batched(st["batch"], st["vm"], st["va"], st["P"], st["Q"], st["J"])
        return st["P"], st["Q"], st["J"]
    if kind == "loss_grad":
        loss = pfgrid.MismatchLoss.apply(st["batch"], *st["leaves"], *st["fixed"], *st["data"])
        return (loss.detach(),) + torch.autograd.grad(loss, st["leaves"])
    if kind == "adjoint":
        pfgrid.adjoint_elementwise(st["batch"], st["vm"], st["va"], *st["data"], *st["out"])
        return tuple(st["out"])
    if kind == "newton_step":
        pfgrid.jac_reduced(grid, "elementwise", st["vm"], st["va"], *st["spec"], st["F"], st["Jr"])
        pfgrid.jac_reduced_solve(grid, st["Jr"], st["F"], st["dx"])
        return st["F"], st["Jr"], st["dx"]
    st["vm"].copy_(st["vm0"])
    st["va"].copy_(st["va0"])
    ok, iterations, _ = pfgrid.powerflow_newton(grid, "elementwise", st["vm"], st["va"], *st["spec"], tol=1e-10)
    return ok, iterations, st["vm"], st["va"]


def work(case):
    """Bytes: parameters of every branch and bus and the states in, results out, once.  Operations: those of the
    methods in plain FP64 (12 per branch terminal and 16 per bus for injections and Jacobian by the element-wise
    method, 16 per admittance entry and per bus by the Ybus method, an FMA counted as two)."""
    kind, nb, nl, S = case["kind"], case["nb"], case["nl"], case["nscen"]
    nnz = nb + 2 * nl
    grid = 48 * nl + 16 * nb
    if kind in ("jac", "host", "n1"):
        return dict(bytes=grid + S * (32 * nb + 32 * nnz), flops=2 * S * (24 * nl + 16 * nb))
    if kind == "inj":
        return dict(bytes=grid + 32 * nb, flops=2 * (16 * nl + 8 * nb))
    if kind in ("ybus_jac", "n1_ybus"):
        return dict(bytes=20 * nnz + 4 * nb + S * (32 * nb + 32 * nnz), flops=2 * S * (16 * nnz + 16 * nb))
    if kind == "ybus_inj":
        return dict(bytes=20 * nnz + 36 * nb, flops=2 * (6 * nnz + 6 * nb))
    if kind in ("loss_grad", "adjoint"):
        return dict(bytes=grid + 32 * nb + 32 * nl + S * 32 * nb, flops=2 * S * (2 * 32 * nl + 22 * nb + 48 * nl))
    # a Newton step: the reduced system out and in again, and about 1.5 times its entries of factor; 4 updates per entry
    steps = 1 if kind == "newton_step" else 3
    entries = int((2 - case["pv"]) ** 2 * nnz)
    return dict(bytes=steps * (grid + 32 * nb + 16 * entries + 24 * entries + 32 * nb),
                flops=2 * steps * (24 * nl + 16 * nb + 6 * entries))


# ------------------------------------------------------------------ 64-bit values of the outputs, plain torch ----

def _targets(gr):
    """P and Q of the grid's second state, summed on the host in one order: the same at every call."""
    P, Q = _powers({k: torch.from_numpy(gr[k]) for k in PARAMS}, *(torch.from_numpy(gr[k]) for k in ("f", "t", "vm2", "va2")))
    return _dev(P.numpy()), _dev(Q.numpy())


def _powers(p, f, t, vm, va):
    """P and Q of one state from the branch parameters p and ends f, t, differentiable."""
    f, t = f.long(), t.long()
    c, s = torch.cos(va[f] - va[t] - p["shift"]), torch.sin(va[f] - va[t] - p["shift"])
    vf, vt, im, half = vm[f], vm[t], 1.0 / p["tap"], 0.5 * p["bsh"]
    w = vf * vt * im
    Pf = vf * vf * im * im * p["g"] - w * (p["g"] * c + p["b"] * s)
    Qf = -vf * vf * im * im * (p["b"] + half) - w * (p["g"] * s - p["b"] * c)
    Pt = vt * vt * p["g"] - w * (p["g"] * c - p["b"] * s)
    Qt = -vt * vt * (p["b"] + half) + w * (p["g"] * s + p["b"] * c)
    P = (vm * vm * p["gs"]).index_add(0, f, Pf).index_add(0, t, Pt)
    Q = (-vm * vm * p["bs"]).index_add(0, f, Qf).index_add(0, t, Qt)
    return P, Q


def _stamps(gr):
    """Ybus pattern (row, column, row pointer, row lengths) and its stamps (entry, value), one block per end."""
    nb, f, t = gr["nb"], gr["f"].astype(np.int64), gr["t"].astype(np.int64)
    d = np.arange(nb, dtype=np.int64)
    keys = np.unique(np.concatenate([d * nb + d, f * nb + t, t * nb + f]))
    row, col = keys // nb, keys % nb
    rp = np.searchsorted(row, np.arange(nb + 1))
    ys, half = gr["g"] + 1j * gr["b"], 0.5j * gr["bsh"]
    m, rot = gr["tap"], np.exp(1j * gr["shift"])
    at = [np.searchsorted(keys, k) for k in (f * nb + f, t * nb + t, f * nb + t, t * nb + f, d * nb + d)]
    val = [(ys + half) / m**2, ys + half, -ys * rot / m, -ys / rot / m, gr["gs"] + 1j * gr["bs"]]
    return [_dev(x) for x in (row, col, rp, np.diff(rp))], [_dev(x) for x in at], [_dev(x) for x in val]


def _jacobian(pat, at, val, vm, va, out=-1):
    """P, Q and the canonical Jacobian values of one state, without branch `out` (its entries then leave the pattern)."""
    row, col, rp, d = pat
    nb, nnz = len(d), len(row)
    Y = torch.zeros(nnz, dtype=torch.complex128, device=DEV)
    for a, v in zip(at, val):
        v = v.clone()
        if out >= 0 and a is not at[4]:
            v[out] = 0
        Y.index_add_(0, a, v)
    U = torch.polar(torch.ones_like(va), va)
    V = vm * U
    I = torch.zeros(nb, dtype=torch.complex128, device=DEV).index_add_(0, row, Y * V[col])
    S = V * I.conj()
    dv = V[row] * (Y * U[col]).conj()
    dth = -1j * vm[col] * dv
    diag = at[4]
    dv[diag] += I.conj() * U
    dth[diag] += 1j * S
    e = torch.arange(nnz, device=DEV)
    x = [rp[row] + e, rp[row] + e + d[row]]
    keep = torch.ones(nnz, dtype=torch.bool, device=DEV)
    if out >= 0:
        h = at[2][out]
        if int((at[2] == h).sum() + (at[3] == h).sum()) == 1:   # no parallel branch keeps the pair
            keep[h] = keep[at[3][out]] = False
    halves = []
    for a, b in ((dth.real, dv.real), (dth.imag, dv.imag)):
        half, kept = torch.empty(2 * nnz, dtype=torch.float64, device=DEV), torch.empty(2 * nnz, dtype=torch.bool, device=DEV)
        half[x[0]], half[x[1]] = a, b
        kept[x[0]], kept[x[1]] = keep, keep
        halves.append(half[kept])
    return S.real, S.imag, torch.cat(halves), (dth, dv)


def exact(case, seed):
    kind, nb, S = case["kind"], case["nb"], case["nscen"]
    gr = _inputs(case, seed)
    vm, va = _dev(gr["vm"]), _dev(gr["va"])
    f, t, p = _dev(gr["f"]), _dev(gr["t"]), {k: _dev(gr[k]) for k in PARAMS}
    if kind in ("inj", "ybus_inj"):
        return _powers(p, f, t, vm[0], va[0])
    if kind in ("jac", "ybus_jac", "host"):
        return _jacobian(*_stamps(gr), vm[0], va[0])[:3]
    if kind in ("n1", "n1_ybus"):
        st = _stamps(gr)
        got = [_jacobian(*st, vm[s], va[s], int(gr["outage"][s]))[:3] for s in range(S)]
        return tuple(torch.cat(x) for x in zip(*got))
    if kind in ("loss_grad", "adjoint"):
        Ps, Qs = _targets(gr)
        wP, wQ = _dev(gr["wP"]), _dev(gr["wQ"])
        for k in PARAMS[:4]:
            p[k].requires_grad_()
        L, gv, gt, gp = [], [], [], None
        for s in range(S):
            v, a = vm[s].clone().requires_grad_(), va[s].clone().requires_grad_()
            P, Q = _powers(p, f, t, v, a)
            loss = (wP * (P - Ps) ** 2 + wQ * (Q - Qs) ** 2).sum()
            g = torch.autograd.grad(loss, [v, a] + [p[k] for k in PARAMS[:4]])
            L.append(loss.detach())
            gv.append(g[0])
            gt.append(g[1])
            gp = list(g[2:]) if gp is None else [x + y for x, y in zip(gp, g[2:])]
        if kind == "loss_grad":
            return (L[0], gv[0], gt[0], *gp)
        return (torch.stack(L), torch.cat(gv), torch.cat(gt), *gp)
    if kind == "powerflow":
        return None, None, _dev(gr["vm2"]), _dev(gr["va2"])
    Ps, Qs = _targets(gr)
    pat, at, val = _stamps(gr)
    P, Q, _, (dth, dv) = _jacobian(pat, at, val, vm[0], va[0])
    bt = _dev(gr["bustype"])
    pvpq, pq = torch.nonzero((bt == 1) | (bt == 2))[:, 0], torch.nonzero(bt == 1)[:, 0]
    F = torch.cat([(P - Ps)[pvpq], (Q - Qs)[pq]])
    n = len(F)
    th = torch.full((nb,), -1, dtype=torch.long, device=DEV)
    mag = th.clone()
    th[pvpq] = torch.arange(len(pvpq), device=DEV)
    mag[pq] = len(pvpq) + torch.arange(len(pq), device=DEV)
    row, col = pat[0], pat[1]
    r = torch.cat([th[row], th[row], mag[row], mag[row]])
    c = torch.cat([th[col], mag[col], th[col], mag[col]])
    x = torch.cat([dth.real, dv.real, dth.imag, dv.imag])
    k = (r >= 0) & (c >= 0)
    r, c, x = r[k], c[k], x[k]
    o = torch.argsort(c * n + r)
    dx = None
    if n <= 5000:   # a dense solve
        A = torch.zeros(n, n, dtype=torch.float64, device=DEV)
        A[r, c] = x
        dx = torch.linalg.solve(A, F)
    return F, x[o], dx
