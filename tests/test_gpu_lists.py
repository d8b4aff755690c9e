"""Tables of graphs whose list lengths sit at the edges of the build passes'
classes: groups of 8, 16 and 32 lanes, a warp, a block in its counting, sorting
and merging forms; empty lists, and lists whose neighbours all have degree 1
(weight zero).  Every table against the oracle, with few and with many records
per warp (the classes are walked 8 or, from 2^18 vertices, 32 records at a
time), in the shared launches of small graphs and in the separate ones."""
from __future__ import annotations

import numpy as np
import pytest

import synth
import paper_1509_08089_gb300 as moss
import test_gpu_min as M
import test_gpu_parity as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EDGES = [1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 1023, 1024, 1025]


def edge_lists(n, more=0):
    """`more` random edges among the pool."""
    rng = np.random.default_rng(5)
    ids = rng.permutation(n)
    pool = ids[:2000]
    at = 2000
    edges = []
    for d in EDGES:
        for _ in range(3):
            edges += [(int(ids[at]), int(x)) for x in rng.choice(pool, d, replace=False)]
            at += 1
    for leaves in (1, 5, 8, 32, 33, 256, 257):     # stars of their own: weight zero at the centre
        edges += [(int(ids[at]), int(x)) for x in ids[at + 1:at + 1 + leaves]]
        at += 1 + leaves
    edges += zip(rng.choice(pool, more), rng.choice(pool, more))
    return synth.from_edges(n, edges)              # the other vertices stay isolated


SIZES = {
    "n4k": (4_001,), "n16383": ((1 << 14) - 1,), "n16384": (1 << 14,), "n262k": ((1 << 18) + 5,),
    "slots_below": (4_001, 110_000), "slots_above": (4_001, 140_000),      # around 2^18 slots
}


def test_slot_sizes_straddle_the_limit():
    below, above = (len(edge_lists(*SIZES[k])[1]) for k in ("slots_below", "slots_above"))
    assert below <= 1 << 18 < above


@pytest.fixture(params=SIZES, scope="module")
def name(request):
    for mod in (P, M):
        mod.GRAPHS[request.param] = lambda: edge_lists(*SIZES[request.param])
    yield request.param
    for mod in (P, M):
        mod.GRAPHS.pop(request.param)
        hit = mod._cache.pop(request.param, None)
        if hit:
            hit[-1].close()


def test_tables_at_the_class_edges(name):
    P.test_tables_bit_exact(name)


def test_min_tables_at_the_class_edges(name):
    M.test_min_tables_bit_exact(name)


@pytest.mark.parametrize("where", ["host", "device", "device32"])
@pytest.mark.parametrize("order", [moss.ORDER_INPUT, moss.ORDER_DEGREE])
def test_small_loads_from_host_and_device(where, order):
    rp, col = edge_lists(4_001)
    ref = moss.Graph(rp, col, order=order)
    if where != "host":
        rp = torch.from_numpy(rp.astype(np.int64 if where == "device" else np.int32)).cuda()
        col = torch.from_numpy(col.view(np.int32)).cuda()
    with moss.Graph(rp, col, order=order) as g:
        a, b = ref.estimate(5, 100_000, 3), g.estimate(5, 100_000, 3)
        assert np.array_equal(a["hits"], b["hits"]) and np.array_equal(a["est"], b["est"])
    ref.close()
