"""The loss sums carry few float32 roundings: a constant |x - y| sums to itself."""
import pytest

torch = pytest.importorskip("torch")

from paper_2503_18402_gb300 import capi  # noqa: E402

pytestmark = pytest.mark.gpu

# three additions in a round, two of the compensated sum, six of the block's tree:
# at most eleven roundings of 2^-24 each, and the result's own
BOUND = 12 * 2.0 ** -24


@pytest.mark.parametrize("V,W,H", [(1, 2000, 1300), (1, 1237, 822), (16, 309, 205), (1, 150, 100), (1, 61, 33), (16, 40, 1001)])
@pytest.mark.parametrize("d", [0.12218045443296432, 0.9364661574363708])
def test_constant_difference(V, W, H, d):
    x = torch.full((V * 3 * W * H,), d, dtype=torch.float32, device="cuda")
    y = torch.zeros_like(x)
    sizes = [(W, H)] * V
    dL, loss = torch.empty_like(x), torch.zeros(V + 1, device="cuda")
    ws = torch.empty(capi.dg_ssim_workspace_size(sizes), dtype=torch.uint8, device="cuda")
    capi.dg_loss_l1_dssim(x, y, sizes, 0.0, dL, loss, ws, ws.numel())
    want = float(x[0].double())
    assert ((loss.double() - want).abs() <= BOUND * want).all()
