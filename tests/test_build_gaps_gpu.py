"""Graphs in which long runs of vertices have no lower (or no upper) neighbour: the built structure
and the time of the build, which must not depend on where such runs lie."""
import time

import numpy as np
import pytest

import paper_1209_6308_gb300 as tc
from test_build_gpu import reference

pytestmark = pytest.mark.gpu


def pairs(n):
    """(i, i + n/2): the first half has no lower neighbour, the second no upper one."""
    i = np.arange(n // 2)
    return i, i + n // 2


def bipartite(left, degree):
    """Left vertices first, each with `degree` right ones, a right one with about half as many."""
    s = np.repeat(np.arange(left), degree)
    return s, left + (np.arange(left * degree) * 7919) % (2 * left)


def islands(n):
    """Pairs, then a run of vertices without any, then a triangle, then another run."""
    i = np.arange(0, n // 4, 2)
    t = n // 2
    return np.concatenate([i, [t, t + 1, t + 2]]), np.concatenate([i + 1, [t + 1, t + 2, t]])


@pytest.mark.parametrize("n,arcs", [(2, pairs(2)), (3, pairs(3)), (4096, pairs(4096)), (70_000, pairs(70_000)),
                                    (30_003, bipartite(10_001, 8)), (999, bipartite(333, 1)), (50_000, islands(50_000))])
@pytest.mark.parametrize("swap", [False, True])
def test_structure_with_runs_of_empty_rows(n, arcs, swap):
    s, d = (np.asarray(a, np.uint32) for a in (arcs[::-1] if swap else arcs))
    off, adj, new, loops, dups = reference(n, s.astype(np.int64), d.astype(np.int64))
    with tc.Graph.from_arcs(n, s, d) as g:
        o, a, p = tc.tc_graph_export_csr(g.handle)
        np.testing.assert_array_equal(p, new)
        np.testing.assert_array_equal(o, off)
        np.testing.assert_array_equal(a, adj)
        forms = [g.census(options={"algo": k}) for k in (0, 1, 2)]
        assert forms[0] == forms[1] == forms[2]


def test_time_of_a_build_with_long_runs():
    """Five million disjoint pairs with the smaller ends first or anywhere are the same work for the sorts
    and more even rows when in order: not slower, with half again for the clock's noise."""
    import torch
    n = 10_000_000
    i = torch.arange(n // 2, dtype=torch.int32, device="cuda")
    p = torch.randperm(n, device="cuda", generator=torch.Generator("cuda").manual_seed(1)).to(torch.int32)
    inputs = {"in_order": (i, i + n // 2), "anywhere": (p[: n // 2].contiguous(), p[n // 2:].contiguous())}
    best = dict.fromkeys(inputs, float("inf"))
    for _ in range(6):
        for name, (s, d) in inputs.items():
            torch.cuda.synchronize()
            t = time.perf_counter()
            tc.Graph.from_arcs(n, s, d).close()
            best[name] = min(best[name], time.perf_counter() - t)
    assert best["in_order"] <= 1.5 * best["anywhere"], best
