"""The two forms of the loss kernels: tiles for small or narrow images, strips of 128
columns in segments of 32 or 64 rows for the rest.  Strips at the edges of their
columns, segments and rounds against the oracle, batches on either side of the
line between the forms, and the gradient bits of both."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2503_18402_gb300 import capi  # noqa: E402
from tests.test_gpu_ssim import _check  # noqa: E402

pytestmark = pytest.mark.gpu


def form(sizes):
    """The library's rule: 0 for tiles, else the rows of a strip's segment."""
    up = lambda a, b: -(-a // b)  # noqa: E731
    strips = lambda rows: sum(3 * up(w, 128) * up(h, rows) for w, h in sizes)  # noqa: E731
    rows = 64 if strips(64) >= 760 else 32
    tiles = sum(3 * up(w, 32) * up(h, 32) for w, h in sizes)
    plain, padded = sum(w * h for w, h in sizes), sum(128 * up(w, 128) * h for w, h in sizes)
    strip_rows = sum(3 * up(w, 128) * (h + 10 * up(h, rows)) for w, h in sizes)
    return 0 if padded * 2 > plain * 3 or tiles <= 2432 or 23 * tiles < 2 * strip_rows else rows


def _pair(rng, W, H):
    x = rng.random((3, H, W))
    return x, np.clip(x + 0.2 * rng.normal(size=x.shape), 0, 1)


@pytest.mark.parametrize("V,W,H,want", [
    (16, 384, 191, 32), (16, 383, 192, 32), (16, 384, 193, 32), (16, 256, 288, 32),
    (16, 512, 255, 64), (16, 511, 256, 64), (16, 510, 257, 64), (3, 1024, 511, 32), (4, 1024, 511, 64),
    (16, 200, 120, 0), (16, 129, 300, 0), (16, 90, 1000, 0), (16, 64, 1030, 0),
])
def test_forms_against_the_oracle(V, W, H, want):
    rng = np.random.default_rng(V + W + H)
    pairs = [_pair(rng, W, H) for _ in range(V)]
    assert form([(W, H)] * V) == want
    _check([p[0] for p in pairs], [p[1] for p in pairs])


@pytest.mark.parametrize("W,H", [(512, 256), (383, 192), (500, 257)])
def test_both_forms_give_the_same_gradient_bits(W, H):
    """One view alone (tiles) and among 16 (strips, whose gradient carries 1/16)."""
    rng = np.random.default_rng(W)
    x, y = (torch.from_numpy(rng.random((16, 3, H, W)).astype(np.float32)).cuda() for _ in range(2))
    assert form([(W, H)]) == 0 and form([(W, H)] * 16) > 0

    def run(a, b, n):
        sizes = [(W, H)] * n
        dL, loss = torch.empty_like(a), torch.zeros(n + 1, device="cuda")
        ws = torch.empty(capi.dg_ssim_workspace_size(sizes), dtype=torch.uint8, device="cuda")
        capi.dg_loss_l1_dssim(a, b, sizes, 0.2, dL, loss, ws, ws.numel())
        return dL, loss

    dL, loss = run(x, y, 16)
    for v in (0, 7, 15):
        d1, l1 = run(x[v].contiguous(), y[v].contiguous(), 1)
        assert torch.equal(dL[v] * 16, d1)
        assert abs(float(l1[0]) - float(loss[v])) <= 2e-6 * float(l1[0])
