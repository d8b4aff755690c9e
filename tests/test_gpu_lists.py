"""Tables of graphs whose list lengths sit at the edges of the build passes'
classes: groups of 8, 16 and 32 lanes, a warp, a block in its counting, sorting
and merging forms; empty lists, and lists whose neighbours all have degree 1
(weight zero).  Every table against the oracle, with few and with many records
per warp (the classes are walked 8 or, from 2^18 vertices, 32 records at a
time)."""
from __future__ import annotations

import numpy as np
import pytest

import synth
import test_gpu_min as M
import test_gpu_parity as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EDGES = [1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 1023, 1024, 1025]


def edge_lists(n):
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
    return synth.from_edges(n, edges)              # the other vertices stay isolated


SIZES = {"edges_n4k": 4_001, "edges_n262k": (1 << 18) + 5}


@pytest.fixture(params=SIZES, scope="module")
def name(request):
    for mod in (P, M):
        mod.GRAPHS[request.param] = lambda: edge_lists(SIZES[request.param])
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
