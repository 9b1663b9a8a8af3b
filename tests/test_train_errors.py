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
