"""The hashed edge set has two to four slots per edge above 2^21 list entries
(four to eight below, and behind the filter): the same samples as list search
where the density changes, where it is highest, and after a change of probe."""
from __future__ import annotations

import numpy as np
import pytest

import synth
import paper_1509_08089_gb300 as moss

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MASK = (1 << 4) | (1 << 5) | moss.TABLES_4MIN


def circulant(n, d):
    """n vertices, each joined to the d / 2 before and after it: n d entries, many triangles."""
    step = np.concatenate([np.arange(-(d // 2), 0), np.arange(1, d // 2 + 1)])
    col = np.sort((np.arange(n)[:, None] + step) % n, axis=1).astype(np.uint32)
    return np.arange(n + 1, dtype=np.int64) * d, col.reshape(-1)


GRAPHS = {
    "at the line": lambda: circulant(1 << 17, 16),          # 2^21 entries: still the roomy set
    "above it": lambda: circulant((1 << 17) + 1, 16),       # 2^21 + 16: half the buckets
    "densest": lambda: circulant((1 << 18) - 1, 16),        # two slots an edge
    "power law": lambda: synth.chung_lu(270_000, 2.3, 14.0, 5000.0, seed=4),
}


@pytest.mark.parametrize("name", GRAPHS)
def test_hashed_samples_equal_searched_ones(name):
    rp, col = GRAPHS[name]()
    K = 200_003
    got = {}
    # each first probe builds the set at its own size; a later one keeps it
    for first, second in ((moss.PROBE_SEARCH, moss.PROBE_HASH), (moss.PROBE_FILTER, moss.PROBE_HASH),
                          (moss.PROBE_HASH, moss.PROBE_FILTER)):
        with moss.Graph(rp, col, k_mask=MASK, probe=first) as g:
            for probe, method in [(p, m) for p in (first, second) for m in range(4)]:
                if probe == second and method == 0:
                    g.set_probe(probe)
                cls = torch.empty(K, dtype=torch.uint8, device="cuda")
                verts = torch.empty(K * 5, dtype=torch.int32, device="cuda")
                moss.moss_sample_records(g.handle, method, 7, K, 11, cls, verts)
                n = 5 if method in (1, 2) else 4
                new = (cls.cpu(), verts.view(K, 5)[:, :n].cpu())
                for a, b in zip(got.setdefault(method, new), new):
                    assert torch.equal(a, b), (probe, method)
