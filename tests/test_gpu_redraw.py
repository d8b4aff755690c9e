"""Path-5's redraws take windows of the deferral bitmap whose width follows the
launch's size: counts and records are the oracle's at the sizes where windows,
rounds of 32 and the last partial words begin and end."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
import paper_1509_08089_gb300 as moss

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WORD_EACH = 152 * 5 * 8 * 32    # ids up to which every warp of the redraw launch has at most one word
SIZES = [1, 31, 33, 1025, WORD_EACH, WORD_EACH + 1, 2 * WORD_EACH - 31, 3 * WORD_EACH + 7]


@pytest.mark.parametrize("probe", [moss.PROBE_SEARCH, moss.PROBE_HASH, moss.PROBE_FILTER])
@pytest.mark.parametrize("rng", [moss.RNG_SPLITMIX64, moss.RNG_PHILOX4X32])
@pytest.mark.parametrize("name", ["complete5", "cl_n20k"])   # 1 of 4 first pairs collides; a few of 100
def test_redraws_at_window_edges(name, rng, probe):
    rp, col = synth.complete(5) if name == "complete5" else synth.chung_lu(20_000, 2.2, 12.0, 900.0, seed=3)
    n = max(SIZES)
    with moss.Graph(rp, col, probe=probe, rng=rng) as g:
        og = oracle.OracleGraph(rp, col)
        _, ocls, overts = og.run(oracle.PATH5, 9, n, record=True, rng=rng)
        out = torch.zeros(22, dtype=torch.int64, device="cuda")
        for K in SIZES:
            moss.moss_sample_counts(g.handle, oracle.PATH5, 0, K, 9, out)
            assert np.array_equal(out.cpu().numpy(), np.bincount(ocls[:K], minlength=22)), K
        cls = torch.empty(n, dtype=torch.uint8, device="cuda")
        verts = torch.empty(n * 5, dtype=torch.int32, device="cuda")
        moss.moss_sample_records(g.handle, oracle.PATH5, 0, n, 9, cls, verts)
        assert np.array_equal(cls.cpu().numpy(), ocls)
        assert np.array_equal(verts.cpu().numpy().view(np.uint32).reshape(n, 5), overts)
