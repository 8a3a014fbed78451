"""Device memory a build holds at its peak, by the library's pool (found through a graph's list)."""
import ctypes

import pytest

import paper_1209_6308_gb300 as tc

pytestmark = pytest.mark.gpu

POINTER_ATTRIBUTE_MEMPOOL_HANDLE, MEMPOOL_ATTR_USED_MEM_HIGH = 17, 8   # cuda.h


def test_peak_of_a_build():
    """Sorting both directions of every pair took 52 B per pair and 40 B per vertex beyond the arcs; sorting
    one direction must not take more, also with the sums and tickets beside the arrays (a MiB)."""
    import torch
    cuda = ctypes.CDLL("libcuda.so.1")
    n, k = 1 << 20, 32                      # x -> x + 1 .. x + 32 (mod n): every arc a pair of its own
    x = torch.arange(n, device="cuda", dtype=torch.int64).repeat_interleave(k)
    d = ((x + 1 + torch.arange(k, device="cuda").repeat(n)) % n).int()
    s = x.int()
    del x
    pool, high = ctypes.c_void_p(), ctypes.c_uint64()
    with tc.Graph.from_arcs(3, s[:2].clone(), d[:2].clone()) as g:
        _, adj, _ = tc.tc_graph_device_csr(g.handle)
        assert cuda.cuPointerGetAttribute(ctypes.byref(pool), POINTER_ATTRIBUTE_MEMPOOL_HANDLE, ctypes.c_uint64(adj)) == 0
    torch.cuda.synchronize()
    assert cuda.cuMemPoolSetAttribute(pool, MEMPOOL_ATTR_USED_MEM_HIGH, ctypes.byref(ctypes.c_uint64(0))) == 0
    cuda.cuMemPoolGetAttribute(pool, 7, ctypes.byref(high))
    before = high.value
    tc.Graph.from_arcs(n, s, d).close()
    assert cuda.cuMemPoolGetAttribute(pool, MEMPOOL_ATTR_USED_MEM_HIGH, ctypes.byref(high)) == 0
    peak, pairs = high.value - before, n * k
    assert 28 * pairs < peak <= 52 * pairs + 40 * n + (1 << 20), (peak, pairs, peak / pairs)
