"""Which filtered calls are grouped follows the list entries, the heavy columns
of the vertex table and the ids; on either side of each line the counts are those
of the ungrouped sampler (moss_sample_counts_noalloc)."""
from __future__ import annotations

import numpy as np
import pytest

import synth
import paper_1509_08089_gb300 as moss

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MASK = (1 << 4) | (1 << 5) | moss.TABLES_4MIN


def counts(fn, g, method, first, count):
    out = torch.full((22,), -1, dtype=torch.int64, device="cuda")
    fn(g.handle, method, first, count, 9, out)
    return out.cpu().numpy()


@pytest.mark.parametrize("order", [moss.ORDER_INPUT, moss.ORDER_DEGREE])
@pytest.mark.parametrize("split", [6, 26])     # few heavy columns; more than 4,096
def test_counts_on_both_sides_of_the_lines(split, order):
    rp, col = synth.chung_lu(20_000, 2.2, 12.0, 900.0, seed=3)
    with moss.Graph(rp, col, k_mask=MASK, probe=moss.PROBE_FILTER, order=order, vsplit=split) as g:
        for method in range(4):
            heavy = moss.moss_vertex_levels(g.handle, method)[0]
            assert method == 3 or (0 < heavy <= 4096 if split == 6 else heavy > 4096)
            for count in ((1 << 22) - 1, 1 << 22, (1 << 23) + 77, (1 << 24) + 77):
                got = counts(moss.moss_sample_counts, g, method, 5, count)
                assert np.array_equal(got, counts(moss.moss_sample_counts_noalloc, g, method, 5, count)), (method, count)
                assert method == 3 or got.sum() == count
