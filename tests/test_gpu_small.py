"""Small estimates draw both sub-methods in one launch and sum, finalize and
return in another; their hits and estimates are those of the separate calls
(moss_sample_counts, moss_finalize) at the sizes where the route changes."""
from __future__ import annotations

import numpy as np
import pytest

import synth
import paper_1509_08089_gb300 as moss

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MASK = (1 << 4) | (1 << 5) | moss.TABLES_4MIN
K5_MOST, MIX_MOST = 1 << 19, 1 << 16     # ids per sub-method up to which both share a launch

GRAPHS = {
    "complete5": lambda: synth.complete(5),                                # Path-5 falls back often
    "star9": lambda: synth.star(9),                                        # no 3-path: every sub-method draws nothing
    "cl_n2k": lambda: synth.workload("cl_n2k"),
    "cl_n20k": lambda: synth.chung_lu(20_000, 2.2, 12.0, 900.0, seed=3),   # two-level vertex tables
}


def counts(g, method, K, seed):
    out = torch.zeros(22, dtype=torch.int64, device="cuda")
    if K:
        moss.moss_sample_counts(g.handle, method, 0, K, seed, out)
    return out.cpu().numpy().astype(np.uint64)


def check(r, g, k, mix, methods, K, seed):
    gamma = list(g.stats().gamma_d)
    K = [n if gamma[m] > 0 else 0 for m, n in zip(methods, K)]
    hits = np.zeros((2, 22), dtype=np.uint64)
    for i, m in enumerate(methods):
        hits[i] = counts(g, m, K[i], seed)
    assert np.array_equal(r["hits"], hits)
    f = moss.result_dict(moss.moss_finalize_min(g.handle, K, hits) if mix else moss.moss_finalize(g.handle, k, K, hits))
    for name in ("K", "est", "var", "lam", "conc", "triangles", "triangles_var"):
        assert np.array_equal(np.asarray(r[name]), np.asarray(f[name]), equal_nan=True), name


@pytest.mark.parametrize("probe", [moss.PROBE_SEARCH, moss.PROBE_HASH, moss.PROBE_FILTER])
@pytest.mark.parametrize("rng", [moss.RNG_SPLITMIX64, moss.RNG_PHILOX4X32])
@pytest.mark.parametrize("name", GRAPHS)
def test_small_estimates_equal_the_separate_calls(name, rng, probe):
    rp, col = GRAPHS[name]()
    with moss.Graph(rp, col, k_mask=MASK, probe=probe, rng=rng) as g:
        for B in (0, 1, 2, 255, 257, 100_001):
            check(g.estimate(5, B, 4), g, 5, False, (1, 2), (B // 2, B - B // 2), 4)
            check(g.estimate_min(B, B // 3, 4), g, 4, True, (0, 3), (B, B // 3), 4)
            check(g.estimate(4, B, 4), g, 4, False, (0,), (B,), 4)


@pytest.mark.parametrize("over", [0, 1])
def test_estimates_across_the_size_limit(over):
    rp, col = GRAPHS["cl_n2k"]()
    with moss.Graph(rp, col, k_mask=MASK) as g:
        K = K5_MOST + over
        check(g.estimate(5, 2 * K, 8), g, 5, False, (1, 2), (K, K), 8)
        K = MIX_MOST + over
        check(g.estimate_min(K, K, 8), g, 4, True, (0, 3), (K, K), 8)
        check(g.estimate_min(3, K, 8), g, 4, True, (0, 3), (3, K), 8)


def test_finalize_takes_host_and_device_counts():
    rp, col = GRAPHS["cl_n2k"]()
    with moss.Graph(rp, col) as g:
        r = g.estimate(5, 50_000, 1)
        K = np.asarray(r["K"], dtype=np.uint64)
        dev = torch.from_numpy(r["hits"].astype(np.int64)).cuda()
        out = moss.moss_result()
        moss._check(moss.load().moss_finalize(g.handle, 5, moss._ptr(K), moss._ptr(dev), moss._stream(None), out))
        assert np.array_equal(moss.result_dict(out)["est"], r["est"])
        cov, r2 = moss.moss_covariance(g.handle, 5, K, r["hits"])
        assert np.array_equal(np.diagonal(cov)[1:], r["var"][1:]) and np.array_equal(cov, cov.T)
        assert np.array_equal(r2["est"], r["est"])


def test_many_graphs_alive_and_released():
    """Results come back through page-locked slots shared by the graphs alive."""
    rp, col = synth.complete(5)
    graphs = [moss.Graph(rp, col) for _ in range(70)]
    ref = graphs[0].estimate(5, 1000, 5)
    for g in graphs[::3]:
        g.close()
    graphs += [moss.Graph(rp, col) for _ in range(5)]
    for g in graphs:
        if g.handle:
            assert np.array_equal(g.estimate(5, 1000, 5)["hits"], ref["hits"])
            g.close()


def test_finalize_beside_a_sampling_call():
    """Counts handed to a finalize on one stream leave those of a sampling call
    in flight on another alone."""
    rp, col = GRAPHS["cl_n20k"]()
    K = 200_000_000
    with moss.Graph(rp, col) as g:
        ref = counts(g, 1, K, 2)
        hits = torch.ones((2, 22), dtype=torch.int64, device="cuda")
        out, res, Ks = torch.zeros(22, dtype=torch.int64, device="cuda"), moss.moss_result(), np.asarray([50, 50], np.uint64)
        side = torch.cuda.Stream()
        torch.cuda.synchronize()
        moss.moss_sample_counts(g.handle, 1, 0, K, 2, out, side)
        moss._check(moss.load().moss_finalize(g.handle, 5, moss._ptr(Ks), moss._ptr(hits), moss._stream(None), res))
        side.synchronize()
        assert np.array_equal(out.cpu().numpy().astype(np.uint64), ref)
        assert (moss.result_dict(res)["hits"] == 1).all()
