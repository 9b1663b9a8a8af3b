"""Selection and placement of the densification at the edges of their tiles
(2048 Gaussians), with budgets of one and of all but one candidate and with
scores that are mostly or all tied (the lower index wins), against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import densify as D  # noqa: E402
from tests.test_gpu_densify import OPTS, _run, _state  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tied", ["few", "most", "all"])
@pytest.mark.parametrize("P", [1, 2047, 2048, 2049, 6200, 70001])
def test_tiles_budgets_and_ties(P, tied):
    g, acc, den = _state(max(P, 98), P)
    g, acc, den = g[:P], acc[:P], den[:P]
    if tied != "few":
        rng = np.random.default_rng(P)
        same = rng.random(P) < (1.0 if tied == "all" else 0.8)
        acc[same], den[same] = np.float32(1.5e-3), np.float32(3.0)
    n_cand = int(D.mark(g, acc, den, np.zeros(P, np.float32), OPTS)["cand"].sum())
    for budget in sorted({0, 1, n_cand // 3, n_cand - 1, n_cand}):
        if 0 <= budget <= n_cand:
            frac = (budget + 0.5) / n_cand if n_cand else 0.0
            got_cand, n_sel = _run(g, acc, den, frac, 3)
            assert got_cand == n_cand and n_sel == budget
