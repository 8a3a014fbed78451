"""The triangle walk over 16-bit lists, tables and warp hashes (walk16.cu): exact counts where its
id windows, table slots and degree bounds meet.  Counts are whole numbers: no tolerance."""
import numpy as np
import pytest

import graphgen
import paper_1209_6308_gb300 as tc

pytestmark = pytest.mark.gpu


def arcs_of(lo, hi, seed):
    """Each pair (lo, hi) as one arc either way or both, a third each."""
    kind = np.random.default_rng(seed).integers(0, 3, len(lo))
    s = np.concatenate([lo[kind != 1], hi[kind != 0]]).astype(np.uint32)
    d = np.concatenate([hi[kind != 1], lo[kind != 0]]).astype(np.uint32)
    return s, d


def circulant(n, offsets):
    """x ~ x + o (mod n): every degree is 2 len(offsets), so the relabelling keeps the ids."""
    x = np.arange(n, dtype=np.int64)
    lo = np.repeat(x, len(offsets))
    hi = (lo + np.tile(np.asarray(offsets, np.int64), n)) % n
    return lo, hi


@pytest.mark.parametrize("n,p", [(2400, 0.5), (6000, 0.1)])
def test_dense_graphs_match_the_suffix_form(n, p):
    n, s, d = graphgen.gnp(n, p, seed=n)
    with tc.Graph.from_arcs(n, s, d) as g:
        st = g.stats()
        assert st["sum_tri_walk"] >= max(64 * st["e_sym"], 7 << 26)     # the form under test
        want = g.census(options={"algo": tc.TC_ALGO_SUFFIX})
        for opts in ({}, {"warp_max_deg": 16}, {"chunk_entries": 8192}, {"item_work": 256}, {"ctas_per_sm": 1}):
            assert g.census(options={"algo": tc.TC_ALGO_TRIANGLE, **opts}) == want


# slot: ids modulo 16384 of the table of one vertex's lower neighbours; 8 multiples of 16384 collide
@pytest.mark.parametrize("name,n,offsets", [
    ("window_edges", 70_000, [1, 2, 3, 5] + [32_766, 32_767, 32_768, 32_769] + list(range(100, 260))),
    ("last_window", 132_000, [1, 2, 4] + [32_768 * k + j for k in (1, 2, 3) for j in (-1, 0, 1)] + list(range(300, 430))),
    ("shared_slots", 140_000, [r + 16_384 * k for r in range(1, 18) for k in range(8)]),
    ("slots_overflow", 140_000, [r + 16_384 * k for r in range(1, 41) for k in range(8)]),
])
def test_regular_graphs_match_the_suffix_form(name, n, offsets):
    lo, hi = circulant(n, [o for o in offsets if o < n // 2] + [n // 2 - 1 - i for i, o in enumerate(offsets) if o >= n // 2])
    s, d = arcs_of(lo, hi, seed=len(name))
    with tc.Graph.from_arcs(n, s, d) as g:
        st = g.stats()
        assert st["sum_tri_walk"] >= max(64 * st["e_sym"], 7 << 26)
        assert g.census(options={"algo": tc.TC_ALGO_TRIANGLE}) == g.census(options={"algo": tc.TC_ALGO_SUFFIX})
        grid = sum(np.array(shard) for shard in _shards(g, 3))
        assert list(grid[1:]) == g.census(options={"algo": tc.TC_ALGO_TRIANGLE})[1:]


def _shards(g, world):
    import torch
    out = torch.zeros(16, dtype=torch.int64, device="cuda")
    for r in range(world):
        tc.tc_census_shard(g.handle, out, r, world, options={"algo": tc.TC_ALGO_TRIANGLE})
        yield out.cpu().tolist()


def test_captured_census_planned_by_another_call():
    """No census has made the 16-bit lists yet: the captured one counts without them."""
    torch = pytest.importorskip("torch")
    n, s, d = graphgen.gnp(2400, 0.5, seed=2400)
    opts = {"algo": tc.TC_ALGO_TRIANGLE}
    with tc.Graph.from_arcs(n, s, d) as g:
        want = g.census(options={"algo": tc.TC_ALGO_SUFFIX})
        tc.tc_census_shard_bounds(g.handle, 1, options=opts)
        out = torch.zeros(16, dtype=torch.int64, device="cuda")
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            tc.tc_census_async(g.handle, out, stream=torch.cuda.current_stream().cuda_stream, options=opts)
        for _ in range(2):
            out.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert out.tolist()[1:] == want[1:]
            assert g.census(options=opts) == want       # makes the lists; the captured launches stay as they were
