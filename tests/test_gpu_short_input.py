"""A CSR array that is shorter than the call says is refused, whether it would be
copied or read in place."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

import synth
import paper_1509_08089_gb300 as moss

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def device_copy(rt, a, nbytes):
    """The first nbytes of a, in an allocation of just that size."""
    p = ctypes.c_void_p()
    assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(nbytes)) == 0
    assert rt.cudaMemcpy(p, ctypes.c_void_p(a.ctypes.data), ctypes.c_size_t(nbytes), 1) == 0
    return p


@pytest.mark.parametrize("order", [moss.ORDER_INPUT, moss.ORDER_DEGREE])
@pytest.mark.parametrize("n", [10_000, 20_000])     # read in place; copied
@pytest.mark.parametrize("short", ["none", "row_ptr", "col"])
def test_short_device_arrays(short, n, order):
    rp, col = synth.chung_lu(n, 2.5, 8.0, 200.0, seed=2)
    rp, col = rp.astype(np.int64), col.astype(np.uint32)
    torch.cuda.init()
    lib, rt, out = moss.load(), ctypes.CDLL("libcudart.so.13"), ctypes.c_void_p()
    a = device_copy(rt, rp, 4096 if short == "row_ptr" else rp.nbytes)
    b = device_copy(rt, col, 4096 if short == "col" else col.nbytes)
    rc = lib.moss_graph_load_csr_order(a, 1, b, len(rp) - 1, len(col), order, 0, None, ctypes.byref(out))
    if short == "none":
        assert rc == 0
        lib.moss_graph_free(out)
    else:
        assert rc != 0 and not out.value
    assert rt.cudaFree(a) == 0 and rt.cudaFree(b) == 0
    with moss.Graph(rp, col, order=order) as g:      # the next call does not report it again
        assert g.stats().nnz == len(col)
