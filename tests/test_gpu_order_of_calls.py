"""What a call reads and writes follows its stream, whatever is in flight: counts
in page-locked memory are read after the copy that fills them, and a call that
is refused or draws nothing leaves the counts of another stream's call alone, and
freeing graphs waits for nobody's work."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

import synth
import paper_1509_08089_gb300 as moss

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MASK = (1 << 4) | (1 << 5) | moss.TABLES_4MIN
LONG = 200_000_000   # samples of a call that is still running when the next one is made


@pytest.fixture(scope="module")
def graph():
    rp, col = synth.chung_lu(20_000, 2.2, 12.0, 900.0, seed=3)
    with moss.Graph(rp, col, k_mask=MASK) as g:
        yield g


@pytest.mark.parametrize("call", ["finalize", "covariance", "finalize_min"])
def test_page_locked_counts_are_read_in_stream_order(graph, call):
    lib, side = moss.load(), torch.cuda.Stream()
    K = np.asarray([500, 500], dtype=np.uint64)
    src = torch.full((2, 22), 3, dtype=torch.int64, device="cuda")
    hits = torch.zeros((2, 22), dtype=torch.int64).pin_memory()
    busy = torch.zeros(22, dtype=torch.int64, device="cuda")
    cov, res = np.zeros((22, 22)), moss.moss_result()
    torch.cuda.synchronize()
    moss.moss_sample_counts(graph.handle, 1, 0, LONG, 2, busy, side)
    with torch.cuda.stream(side):
        hits.copy_(src, non_blocking=True)
    assert not side.query()
    h, s, out = ctypes.c_void_p(hits.data_ptr()), side.cuda_stream, ctypes.byref(res)
    if call == "finalize":
        moss._check(lib.moss_finalize(graph.handle, 5, moss._ptr(K), h, s, out))
    elif call == "covariance":
        moss._check(lib.moss_covariance(graph.handle, 5, moss._ptr(K), h, s, moss._ptr(cov), out))
    else:
        moss._check(lib.moss_finalize_min(graph.handle, moss._ptr(K), h, s, None, out))
    assert (moss.result_dict(res)["hits"] == 3).all()


def refused(g, out):
    for method, first, count in ((-1, 0, 5), (7, 0, 5), (1, 2**64 - 1, 2), (2, 0, 2**63)):
        with pytest.raises(moss.MossError):
            moss.moss_sample_counts(g.handle, method, first, count, 2, out)
    with pytest.raises(moss.MossError):
        g.estimate(4, 2**63, 2)
    with pytest.raises(moss.MossError):
        g.estimate_min(5, 2**63, 2)


def empty(g, out):
    moss.moss_sample_counts(g.handle, 1, 9, 0, 2, out)
    for r in (g.estimate(4, 0, 2), g.estimate(5, 0, 2), g.estimate_min(0, 0, 2)):
        assert not r["hits"].any()
    torch.cuda.current_stream().synchronize()
    assert not out.any()


@pytest.mark.parametrize("other", [refused, empty])
@pytest.mark.parametrize("method", [1, 2])
def test_a_call_that_draws_nothing_leaves_another_streams_counts(graph, method, other):
    def counts(stream=None):
        moss.moss_sample_counts(graph.handle, method, 0, LONG, 2, out, stream)

    out, none = (torch.full((22,), -1, dtype=torch.int64, device="cuda") for _ in range(2))
    counts()
    torch.cuda.synchronize()
    ref = out.clone()
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    counts(side)
    assert not side.query()
    other(graph, none)
    side.synchronize()
    assert torch.equal(out, ref)


def test_freeing_graphs_does_not_wait_for_the_device(graph):
    rp, col = synth.complete(5)
    graphs = [moss.Graph(rp, col) for _ in range(70)]
    out, side = torch.zeros(22, dtype=torch.int64, device="cuda"), torch.cuda.Stream()
    torch.cuda.synchronize()
    moss.moss_sample_counts(graph.handle, 1, 0, 20 * LONG, 2, out, side)
    for g in graphs:
        g.close()
    assert not side.query()
    side.synchronize()
    assert int(out.sum()) == 20 * LONG


def test_calls_of_many_threads(graph):
    """More calls at a time than there are page-locked slots to lend."""
    from concurrent.futures import ThreadPoolExecutor
    rp, col = synth.complete(5)
    graphs = [moss.Graph(rp, col) for _ in range(48)]
    hits = np.ones((2, 22), dtype=np.uint64)
    ref = moss.moss_covariance(graphs[0].handle, 5, np.array([50, 50], np.uint64), hits)

    want = graphs[0].estimate(5, 1000, 5)["hits"]

    def use(g):
        for _ in range(10):
            assert np.array_equal(g.estimate(5, 1000, 5)["hits"], want)
            cov, r = moss.moss_covariance(g.handle, 5, np.array([50, 50], np.uint64), hits)
            assert np.array_equal(cov, ref[0]) and np.array_equal(r["est"], ref[1]["est"])
        return True

    with ThreadPoolExecutor(48) as pool:
        assert all(pool.map(use, graphs))
    for g in graphs:
        g.close()
