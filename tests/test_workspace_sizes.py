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
    counts = _around(1024, 2 * lim, 3 * lim, 5 * lim, 8 * lim, 20 * lim, 1 << 30) + [0, 5, 100000, 3_000_000]
    counts = sorted(set(counts))
    for views in (1, 3, 16):
        for M in (0, 5 * lim, 5 * lim + 1, 4_000_000):
            sizes = [capi.dg_bin_workspace_size(P, views, M) for P in counts]
            assert sizes == sorted(sizes)
        for P in (1000, 3 * lim, 3 * lim + 1, 2_000_000):
            sizes = [capi.dg_bin_workspace_size(P, views, M) for M in counts]
            assert sizes == sorted(sizes)
    for P in counts[:-6]:
        sizes = [capi.dg_bin_workspace_size(P, v, 5 * lim + 1) for v in range(1, 17)]
        assert sizes == sorted(sizes)
