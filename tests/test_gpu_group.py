"""Large sampling calls behind the edge filter are drawn in groups of ids that
share their first vertex; the counts are those of the ungrouped sampler, which
moss_sample_counts_noalloc runs for any size."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
import paper_1509_08089_gb300 as moss

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MASK = (1 << 4) | (1 << 5) | moss.TABLES_4MIN
INPUT_MIN, DEGREE_MIN = 1 << 22, 1 << 24     # ids from which a call is grouped


def counts(fn, g, method, first, count, seed, stream=None):
    out = torch.full((22,), -1, dtype=torch.int64, device="cuda")
    fn(g.handle, method, first, count, seed, out, stream)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def same(g, method, first, count, seed):
    ref = counts(moss.moss_sample_counts_noalloc, g, method, first, count, seed)
    got = counts(moss.moss_sample_counts, g, method, first, count, seed)
    assert np.array_equal(got, ref), (method, first, count, got, ref)
    return got


GRAPHS = {
    "complete6": lambda: synth.complete(6),                       # six groups hold every id; one Path-5 pair in 5 collides
    "cl_n2k": lambda: synth.workload("cl_n2k"),                   # one-level vertex tables
    "cl_n20k": lambda: synth.chung_lu(20_000, 2.2, 12.0, 900.0, seed=3),   # two levels
}


@pytest.mark.parametrize("rng", [moss.RNG_SPLITMIX64, moss.RNG_PHILOX4X32])
@pytest.mark.parametrize("name", GRAPHS)
def test_grouped_counts_equal_the_ungrouped(name, rng):
    rp, col = GRAPHS[name]()
    with moss.Graph(rp, col, k_mask=MASK, probe=moss.PROBE_FILTER, rng=rng) as g:
        for method in range(4):
            # the first grouped size, one below it, a ragged tail
            for first, count in ((0, INPUT_MIN), (77, INPUT_MIN - 1), ((1 << 40) + 5, INPUT_MIN + 8191)):
                same(g, method, first, count, 11 + method)


def test_grouped_counts_equal_the_oracle():
    rp, col = synth.workload("cl_n2k")
    og = oracle.OracleGraph(rp, col)
    with moss.Graph(rp, col, probe=moss.PROBE_FILTER) as g:
        got = counts(moss.moss_sample_counts, g, oracle.PATH5, 0, INPUT_MIN + 1, 9)
    assert np.array_equal(got.astype(np.uint64), og.run(oracle.PATH5, 9, INPUT_MIN + 1))


def test_grouped_in_degree_order_and_across_chunks():
    rp, col = GRAPHS["cl_n20k"]()
    with moss.Graph(rp, col, k_mask=MASK, probe=moss.PROBE_FILTER, order=moss.ORDER_DEGREE,
                    vsplit=moss.VERTEX_ONE_LEVEL) as g:
        for method in range(4):
            same(g, method, 3, DEGREE_MIN + 1, 5)
            same(g, method, 3, DEGREE_MIN - 1, 5)
    with moss.Graph(rp, col, probe=moss.PROBE_FILTER, order=moss.ORDER_DEGREE) as g:
        got = same(g, oracle.PATH5, 1, (1 << 26) + 12_345, 6)     # two chunks of the deferral bitmap
        assert int(got.sum()) == (1 << 26) + 12_345
        same(g, oracle.T5, 1, DEGREE_MIN + 1, 6)                  # few heavy vertices in degree order: not grouped


def test_capture_takes_the_ungrouped_path():
    """Under stream capture the call allocates nothing and replays."""
    rp, col = synth.workload("cl_n2k")
    with moss.Graph(rp, col, probe=moss.PROBE_FILTER) as g:
        n = INPUT_MIN + 17
        ref = counts(moss.moss_sample_counts, g, oracle.T5, 0, n, 2)
        out = torch.zeros(22, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            moss.moss_sample_counts(g.handle, oracle.T5, 0, n, 2, out)
        for _ in range(2):
            out.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert np.array_equal(out.cpu().numpy(), ref)
