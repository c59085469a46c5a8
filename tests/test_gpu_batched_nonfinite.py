"""Batched injections beside a bus without a finite state: an outage takes its
branch out of the sums whatever the other end holds, as in a grid without it.
"""
import numpy as np
import pytest

from gridcases import random_grid, random_state

pytestmark = pytest.mark.gpu

TOL = 1e-12   # as against the oracle


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("which", ["vm", "va"])
@pytest.mark.parametrize("call", ["elementwise", "ybus"])
def test_outage_beside_a_bad_bus(bad, which, call):
    import torch
    from paper_2302_10736_gb300 import pfgrid as pf
    nb = 400
    gr = random_grid(nb, 540, 4, shift_max=0.2)
    pairs = {}
    for l, (f, t) in enumerate(zip(gr["f"], gr["t"])):
        pairs.setdefault((min(f, t), max(f, t)), []).append(l)
    out = [ls[0] for ls in pairs.values() if len(ls) == 1][:40:5]
    dev = lambda x: torch.tensor(x, dtype=torch.float64, device="cuda")
    S = len(out)
    vm, va = random_state(nb, 6, S)
    for s, l in enumerate(out):
        (vm if which == "vm" else va)[s, gr["t" if s % 2 else "f"][l]] = bad
    batch = pf.batch_create(pf.ybus_build(gr), S, np.array(out, np.int32))
    P, Q = (torch.full((S * nb,), 7.0, dtype=torch.float64, device="cuda") for _ in range(2))
    fn = pf.inj_elementwise_batched if call == "elementwise" else pf.inj_ybus_batched
    fn(batch, dev(vm.ravel()), dev(va.ravel()), P, Q)
    got = [x.cpu().numpy().reshape(S, nb) for x in (P, Q)]
    for s, l in enumerate(out):
        keep = np.arange(gr["nl"]) != l
        one = {k: v[keep] if k in ("f", "t", "g", "b", "bsh", "tap", "shift") else v for k, v in gr.items()}
        one["nl"] = gr["nl"] - 1
        grid = pf.ybus_build(one)
        Pr, Qr = (torch.full((nb,), 7.0, dtype=torch.float64, device="cuda") for _ in range(2))
        (pf.inj_elementwise if call == "elementwise" else pf.inj_ybus)(grid, dev(vm[s]), dev(va[s]), Pr, Qr)
        other = gr["f" if s % 2 else "t"][l]   # the outage's good end
        for x, y in zip(got, (Pr.cpu().numpy(), Qr.cpu().numpy())):
            ok = np.isfinite(y)
            assert np.array_equal(np.isfinite(x[s]), ok), (s, np.flatnonzero(np.isfinite(x[s]) != ok))
            assert np.max(np.abs(x[s][ok] - y[ok])) <= TOL * np.max(np.abs(y[ok]))
        assert np.isfinite(got[0][s, other]) and np.isfinite(got[1][s, other])
