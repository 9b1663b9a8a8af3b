"""A workspace laid out for more records, views or pairs serves fewer (CPU only: the
sizes are host arithmetic)."""
from __future__ import annotations

import pytest


@pytest.fixture(scope="module")
def capi():
    from paper_2503_18402_gb300 import build
    build.build()
    from paper_2503_18402_gb300 import capi as c
    return c


def _around(*limits):
    return sorted({max(0, x + d) for x in limits for d in (-1025, -1, 0, 1, 1025)})


def test_binning_workspace_grows_with_every_count(capi):
    # the counts at which the passes and the record kernel change their block sizes,
    # the look-back words their width, and sizes between
    lim = 152 * 1024
    counts = _around(1024, 2 * lim, 5 * lim // 2, 3 * lim, 5 * lim, 8 * lim, 20 * lim, 1 << 30) + [0, 5, 100000, 3_000_000]
    counts = sorted(set(counts))
    for views in (1, 3, 16):
        for M in (0, 5 * lim, 5 * lim + 1, 4_000_000):
            sizes = [capi.dg_bin_workspace_size(P, views, M) for P in counts]
            assert sizes == sorted(sizes)
        for P in (1000, 5 * lim // 2, 5 * lim // 2 + 1, 2_000_000):
            sizes = [capi.dg_bin_workspace_size(P, views, M) for M in counts]
            assert sizes == sorted(sizes)
    for P in counts[:-6]:
        sizes = [capi.dg_bin_workspace_size(P, v, 5 * lim + 1) for v in range(1, 17)]
        assert sizes == sorted(sizes)


def test_loss_workspace_grows_with_every_size(capi):
    import random
    rng = random.Random(1)
    for _ in range(2000):
        big = [(rng.randint(1, 700), rng.randint(1, 700)) for _ in range(rng.choice([1, 1, 2, 3, 16]))]
        small = [(rng.randint(1, w), rng.randint(1, h)) for w, h in big]
        assert capi.dg_ssim_workspace_size(small) <= capi.dg_ssim_workspace_size(big), (small, big)
    # narrow images: at most half as many map values again as pixels, and the block sums
    for w in (1, 5, 33, 129):
        n = w * 60000
        assert capi.dg_ssim_workspace_size([(w, 60000)]) <= 36 * (n + n // 2 + 1) + 24 * (-(-w // 32)) * 1875 + 512
