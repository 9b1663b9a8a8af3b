"""What the trainer does with error words of the library (no GPU: the calls are fakes)."""
from __future__ import annotations

from types import SimpleNamespace

import pytest

pytest.importorskip("torch")

from paper_2503_18402_gb300 import capi  # noqa: E402
from paper_2503_18402_gb300.train import Trainer  # noqa: E402


def _pending(status):
    g = SimpleNamespace(sizes=[(64, 48)], key="k", result=lambda slot: (status, 123))
    return SimpleNamespace(pending=[(g, 0)], M_hint={}, skipped_steps=0, graphs={"k": g})


def test_replayed_steps_tell_overflow_from_failure():
    tr = _pending(capi.DG_OK)
    Trainer._check_pending(tr, keep=0)
    assert tr.skipped_steps == 0 and "k" in tr.graphs
    tr = _pending(capi.DG_ERR_CAPACITY)
    Trainer._check_pending(tr, keep=0)
    assert tr.skipped_steps == 1 and not tr.graphs and tr.M_hint == {(64, 48): 123}
    for code in (capi.DG_ERR_TIMEOUT, capi.DG_ERR_CUDA):
        with pytest.raises(capi.DashGSError) as e:
            Trainer._check_pending(_pending(code), keep=0)
        assert e.value.status == code


def test_a_failed_densification_leaves_the_model(monkeypatch):
    """The library writes an error word where the new count belongs: the trainer
    raises and keeps its count, buffers and statistics."""
    import torch
    from paper_2503_18402_gb300.train import TrainConfig

    P, cap = 5, 12
    buf = [dict(p=torch.ones(59, cap), m=torch.ones(59, cap), v=torch.ones(59, cap)) for _ in range(2)]
    tr = SimpleNamespace(cfg=TrainConfig(), P=P, cap=cap, buf=buf, cur=0, dws=None, dev=torch.device("cpu"),
                         stream=None, acc=torch.ones(cap), den=torch.ones(cap), maxr=torch.ones(cap), sched=None,
                         counts=torch.tensor([4, 2]), P_out=torch.zeros(1, dtype=torch.int64),
                         gen=torch.Generator(), history=[])
    outcome = {}

    def apply(*a):
        tr.P_out.fill_(outcome["P"])

    monkeypatch.setattr(capi, "dg_densify_mark", lambda *a: None)
    monkeypatch.setattr(capi, "dg_densify_apply", apply)
    outcome["P"] = capi.DG_ERR_TIMEOUT
    with pytest.raises(capi.DashGSError) as e:
        Trainer._densify(tr, 600)
    assert e.value.status == capi.DG_ERR_TIMEOUT
    assert tr.P == P and tr.cur == 0 and not tr.history
    assert float(tr.acc.sum()) == cap and float(tr.den.sum()) == cap
    outcome["P"] = 7
    Trainer._densify(tr, 600)
    assert tr.P == 7 and tr.cur == 1 and tr.history[0]["P"] == 7 and float(tr.acc.sum()) == 0
