"""The kernels bench.py claims for a step (device_launches) and the calls it
takes as grouped, worked out from the launch code for each kind of step."""
from __future__ import annotations

import numpy as np
import pytest

import bench


def csr_ends(n, d, d_max):
    """row_ptr of n lists: one of d_max entries, the others of d."""
    deg = np.full(n, d, dtype=np.int64)
    deg[0] = d_max
    return np.concatenate([[0], np.cumsum(deg)])


SMALL, MID, LARGE = csr_ends(2_000, 8, 200), csr_ends(100_000, 20, 4_230), csr_ends(1_200_000, 14, 20_000)


@pytest.mark.parametrize("rp,k,budget,mix,probe,two,two_min,order,grouped,expected", [
    # shared launches (load 4, build 4), both sub-methods in one, finalize
    (SMALL, 5, 100_000, False, "hash", False, False, "input", (), 4 + 4 + 1 + 1),
    (SMALL, 4, 100_000, False, "hash", False, False, "degree", (), 4 + 4 + 4 + 1 + 1),
    # load 8; build: lists up to 256, of 257..2,048 and above, fill, four vertex-table phases after the three of
    # the level split, edge set; T-5, Path-5 and its redraws; finalize
    (MID, 5, 10**8, False, "hash", True, False, "input", (), 8 + 4 + 7 + 1 + 3 + 1),
    # MOSS-4Min: three sort tiers, records, three alias passes, picks, total, four phases (one level)
    (MID, 4, 10**8, True, "hash", True, False, "input", (), 8 + 4 + 7 + 1 + 13 + 2 + 1),
    # behind the filter: the filter and six hub kernels; grouped: draw, scan, placement and sampler a chunk of
    # 2^26 ids, Path-5 its redraws beside them
    (LARGE, 5, 10**9, False, "filter", True, True, "degree", (1, 2), 4 + 8 + 4 + 7 + 1 + 7 + 8 * 4 + 8 * 5 + 1),
    (LARGE, 5, 10**9, False, "filter", True, True, "input", (2,), 8 + 4 + 7 + 1 + 7 + 1 + 8 * 5 + 1),
])
def test_device_launches(rp, k, budget, mix, probe, two, two_min, order, grouped, expected):
    assert bench.device_launches(rp, k, budget, mix, probe, two, two_min, order, grouped) == expected


@pytest.mark.parametrize("m,nnz,heavy,order,least", [
    (0, 7_000_000, 500, "input", None), (0, 14_000_000, 500, "input", 1 << 23), (0, 20_000_000, 0, "input", 1 << 22),
    (1, 7_000_000, 500, "input", None), (1, 14_000_000, 500, "input", 1 << 22), (1, 5_000_000, 0, "input", 1 << 22),
    (2, 7_000_000, 500, "input", 1 << 23), (2, 14_000_000, 500, "input", 1 << 22),
    (3, 7_000_000, 0, "input", 1 << 23), (3, 14_000_000, 0, "input", 1 << 22),
    (0, 14_000_000, 500, "degree", None), (2, 5_000_000, 500, "degree", 1 << 24), (3, 5_000_000, 0, "degree", 1 << 24),
    (0, 24_000_000, 9_000, "degree", None), (0, 68_000_000, 9_000, "degree", 1 << 24),
    (1, 24_000_000, 9_000, "degree", 1 << 24), (2, 16_000_000, 9_000, "degree", None),
])
def test_grouped_calls(m, nnz, heavy, order, least):
    for K in (1 << 21, 1 << 22, 1 << 23, 1 << 24, 10**9):
        assert bench.groups(m, nnz, heavy, K, "filter", order) == (least is not None and K >= least), K
    assert not bench.groups(m, nnz, heavy, 10**9, "hash", order)
