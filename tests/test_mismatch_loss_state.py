"""MismatchLoss keeps the forward pass's values for its backward pass (host only:
the library's calls are replaced by ones that note what they are given).
"""
import types

import pytest

torch = pytest.importorskip("torch")

from paper_2302_10736_gb300 import pfgrid as pf  # noqa: E402

NAMES = ("vm", "va", "g", "b", "bsh", "tap", "shift", "gs", "bs", "Ps", "Qs", "wP", "wQ")


@pytest.mark.parametrize("change", ["none", "data", "set_"])
def test_backward_sees_the_forward_state(monkeypatch, change):
    nb, nl = 3, 2
    size = {k: nl if k in ("g", "b", "bsh", "tap", "shift") else nb for k in NAMES}
    x = {k: torch.full((size[k],), float(i + 1), dtype=torch.float64) for i, k in enumerate(NAMES)}
    for k in NAMES[:6]:
        x[k].requires_grad_()
    seen = []
    note = lambda ts: seen.append([None if t is None else t.clone() for t in ts])
    monkeypatch.setattr(pf, "grid_set_params", lambda grid, *p: note(p))
    monkeypatch.setattr(pf, "loss_elementwise", lambda batch, *a: (note(a[:6]), a[7].fill_(1.0)))

    def adjoint(batch, vm, va, Ps, Qs, wP, wQ, L, *grads, Lbar=None):
        note((vm, va, Ps, Qs, wP, wQ))
        for t in grads:
            t.fill_(float(Lbar))

    monkeypatch.setattr(pf, "adjoint_elementwise", adjoint)
    batch = types.SimpleNamespace(nscen=1, grid=types.SimpleNamespace(nb=nb, nl=nl))
    loss = pf.MismatchLoss.apply(batch, *x.values())
    for k in NAMES:
        new = torch.full_like(x[k], -9.0).detach()
        if change == "data":
            x[k].data = new
        elif change == "set_":
            with torch.no_grad():
                x[k].set_(new)
    (2.0 * loss).backward()
    params, state = seen[:2]
    assert len(seen) == 4
    for then, now in ((params, seen[2]), (state, seen[3])):
        for a, b in zip(then, now):
            assert torch.equal(a, b)
    assert torch.equal(x["vm"].grad, torch.full((nb,), 2.0, dtype=torch.float64))
