"""The autotuner times a tile size only where it changes how the run is cut."""
from __future__ import annotations

import pytest

import synth
import paper_1509_08089_gb300 as moss

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_equal_plans_are_one_candidate():
    # 64 pieces a warp of the whole chip leave pieces of 256 samples, below every candidate
    rp, col = synth.workload("cl_n2k")
    with moss.Graph(rp, col) as g, moss.Batch() as b:
        for seed in range(8):
            b.add(g, 5, 100_000, seed)
        first = b.run()
        assert b.tune() == 1024 and b.tuning()["tile_samples"] == 1024
        for r, q in zip(first, b.run()):
            assert (r["hits"] == q["hits"]).all() and (r["est"] == q["est"]).all()
