"""Targets of a captured step: one concatenation of like images, or copies one by
one; both put the same values at the same places (no GPU needed)."""
from types import SimpleNamespace

import pytest

torch = pytest.importorskip("torch")

from paper_2503_18402_gb300.graphstep import StepGraph  # noqa: E402


@pytest.mark.parametrize("case", ["like", "one", "strided", "float64", "grad", "own_buffer", "short"])
def test_targets_are_placed_in_order(case):
    shapes = [(3, 5, 7)] if case == "one" else [(3, 5, 7), (3, 4, 6), (3, 1, 1)]
    g = torch.Generator().manual_seed(3)
    ts = [torch.rand(s, generator=g) for s in shapes]
    total = sum(t.numel() for t in ts)
    dst = torch.full((total + (5 if case == "short" else 0),), -1.0)
    if case == "strided":
        ts[1] = torch.rand((6, 4, 3), generator=g).permute(2, 1, 0)
    if case == "float64":
        ts[1] = ts[1].double()
    if case == "own_buffer":
        ts[0] = dst[:105].view(3, 5, 7)
    want = torch.cat([t.reshape(-1).float() for t in ts])
    if case == "grad":
        with torch.no_grad():
            StepGraph._copy_targets(SimpleNamespace(target=dst), [ts[0], ts[1].requires_grad_(), ts[2]])
    else:
        StepGraph._copy_targets(SimpleNamespace(target=dst), ts)
    assert torch.equal(dst[:total], want) and bool((dst[total:] == -1).all())


def test_targets_larger_than_the_buffer_are_refused():
    with pytest.raises(RuntimeError):
        StepGraph._copy_targets(SimpleNamespace(target=torch.zeros(10)), [torch.ones(6), torch.ones(6)])
