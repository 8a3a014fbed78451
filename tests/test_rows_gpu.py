"""Kernels that share a warp among short lists (rows.cuh, the packed one-warp walk) and split long
ones over a CTA, at list lengths around their limits.  Counts are whole numbers: no tolerance."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_1209_6308_gb300 as tc

pytestmark = pytest.mark.gpu


def hubs(degrees, first, step):
    """Hubs of the given degrees at caller ids first, first + step, ...; each links the ids around it
    (hubs among them), a third of the links one way, a third the other, a third both."""
    n = 1400
    rng = np.random.default_rng(len(degrees) + first)
    s, d = [], []
    for i, k in enumerate(degrees):
        h = first + step * i
        others = rng.permutation(np.delete(np.arange(n), h))[:k]
        kind = rng.integers(0, 3, k)
        s += [np.full((kind != 1).sum(), h), others[kind != 0]]
        d += [others[kind != 1], np.full((kind != 0).sum(), h)]
    return n, np.concatenate(s).astype(np.uint32), np.concatenate(d).astype(np.uint32)


@pytest.mark.parametrize("degrees", [[31, 32, 33], [255, 256, 257], [224, 287, 289], [511, 513, 1025], [1, 2, 1399]])
@pytest.mark.parametrize("first,step", [(0, 1), (700, 3), (1390, 2)])
def test_lists_around_the_limits(degrees, first, step):
    n, s, d = hubs(degrees, first, step)
    with tc.Graph.from_arcs(n, s, d) as g:
        assert g.census64() == oracle.census64(n, s, d)
        want = oracle.census_bm(n, s, d)
        for algo in (tc.TC_ALGO_SUFFIX, tc.TC_ALGO_TRIANGLE):
            assert g.census(options={"algo": algo}) == want


# degrees about the 32 pairs, 128 lower entries and 32 rows of a pack, and the one-warp tier's bound
@pytest.mark.parametrize("n,p", [(40, 0.9), (70, 0.5), (129, 0.45), (260, 0.12), (700, 0.01), (3000, 0.0006)])
def test_packed_vertices(n, p):
    graphs = [graphgen.gnp(n, p, seed) for seed in (1, 2, 3)]
    want = [oracle.census_bm(*g) for g in graphs]
    handles = [tc.Graph.from_arcs(*g) for g in graphs]
    for warp_max in (16, 64, 128):
        opts = {"algo": tc.TC_ALGO_TRIANGLE, "warp_max_deg": warp_max}
        for h, w in zip(handles, want):
            assert h.census(options=opts) == w
        b = tc.tc_batch_create([h.handle for h in handles], options=opts)
        assert tc.tc_batch_census(b, len(handles)) == want
        tc.tc_batch_destroy(b)


# The bulk sums of a lane are 32 bits wide for 2^31 / n rounds of 32 pairs: with 2^28 vertices, 7.  The
# other vertices have no link, so the compact graph's counts change in the classes of one link only.
@pytest.mark.parametrize("k", [300, 1399])
def test_bulk_sums_of_many_vertices(k):
    n = 1 << 28
    c, s, d = hubs([k, 1399, 1000, 700], 5, 100)
    want = oracle.census_bm(c, s, d)
    pairs = set(zip(s.tolist(), d.tolist()))
    mutual = sum((b, a) in pairs for a, b in pairs) // 2
    want = list(want)
    want[1] += (len(pairs) - 2 * mutual) * (n - c)
    want[2] += mutual * (n - c)
    want[0] = n * (n - 1) * (n - 2) // 6 - sum(want[1:])
    at = np.sort(np.random.default_rng(k).choice(n, c, replace=False)).astype(np.uint32)
    with tc.Graph.from_arcs(n, at[s], at[d]) as g:
        for item_work in (0, 1 << 20):
            assert list(g.census(options={"algo": tc.TC_ALGO_TRIANGLE, "item_work": item_work})) == want
