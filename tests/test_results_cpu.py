"""Unpacking an array of results: the values of result_dict, in memory that a
kept result shares with few others."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

import paper_1509_08089_gb300 as moss


@pytest.mark.parametrize("n", [1, 63, 64, 65, 200])
def test_result_dicts(n):
    arr = (moss.moss_result * n)()
    raw = np.frombuffer(arr, dtype=np.uint8)
    raw[:] = np.random.default_rng(n).integers(0, 64, raw.size)   # (finite doubles)
    got = moss.result_dicts(arr)
    assert len(got) == n
    for r, d in zip(arr, got):
        ref = moss.result_dict(r)
        assert list(d) == list(ref)
        for k in ref:
            assert type(d[k]) is type(ref[k]) and np.array_equal(d[k], ref[k]), k
    raw[:] = 0
    held = {}
    for k, v in got[0].items():
        if isinstance(v, np.ndarray):
            assert v.flags.writeable and v.any()
            while isinstance(v, np.ndarray):
                v = v.base
            held[id(v.obj)] = len(v.obj)
    assert sum(held.values()) <= 64 * ctypes.sizeof(moss.moss_result)
