"""Once a call has made a graph's plan, a census of it only launches: it neither waits for the stream nor
allocates, whichever call made the plan.  Counts are whole numbers: no tolerance."""
import pytest
import torch

import graphgen
import paper_1209_6308_gb300 as tc

pytestmark = pytest.mark.gpu

TRI = {"algo": tc.TC_ALGO_TRIANGLE}


@pytest.fixture(scope="module")
def graph():
    n, s, d = graphgen.gnp(2400, 0.5, seed=2400)
    with tc.Graph.from_arcs(n, s, d) as g:
        want = g.census(options={"algo": tc.TC_ALGO_SUFFIX})
    return n, s, d, want


def _async(g, out, cycles, stream):
    tc.tc_census_async(g.handle, out, stream=stream, options=TRI)


def _shard(g, out, cycles, stream):
    tc.tc_census_shard(g.handle, out, 0, 1, stream=stream, options=TRI)


def _profile(g, out, cycles, stream):
    tc.tc_census_profile(g.handle, out, cycles, stream=stream, options=TRI)


@pytest.mark.parametrize("call", [_async, _shard, _profile])
def test_a_planned_census_does_not_wait(graph, call):
    """The first census of a graph large enough for the 16-bit lists, planned by tc_census_shard_bounds,
    returns while a kernel before it on the stream still runs (half a second)."""
    n, s, d, want = graph
    with tc.Graph.from_arcs(n, s, d) as g:
        st = g.stats()
        assert st["sum_tri_walk"] >= max(64 * st["e_sym"], 7 << 26)
        tc.tc_census_shard_bounds(g.handle, 1, options=TRI)
        out = torch.zeros(16, dtype=torch.int64, device="cuda")
        cycles = torch.zeros(n, dtype=torch.int64, device="cuda")
        stream = torch.cuda.Stream()
        with tc.Graph.from_arcs(n, s, d) as warm:                   # the kernels are loaded
            call(warm, out, cycles, stream.cuda_stream)
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            torch.cuda._sleep(1_000_000_000)
            slept = torch.cuda.Event()
            slept.record(stream)
        call(g, out, cycles, stream.cuda_stream)
        waited = slept.query()
        torch.cuda.synchronize()
        assert not waited
        assert out.tolist()[1:] == want[1:]


def test_captured_census_planned_by_a_call_without_lists(graph):
    """The 64-state census plans this chunk and occupancy but reads no 16-bit lists, and a captured census
    cannot make them: it counts without."""
    n, s, d, want = graph
    opts = {**TRI, "chunk_entries": 1024, "ctas_per_sm": 5}
    with tc.Graph.from_arcs(n, s, d) as g:
        g.census64()
        out = torch.zeros(16, dtype=torch.int64, device="cuda")
        capture = torch.cuda.CUDAGraph()
        with torch.cuda.graph(capture):
            tc.tc_census_async(g.handle, out, stream=torch.cuda.current_stream().cuda_stream, options=opts)
        for _ in range(2):
            out.zero_()
            capture.replay()
            torch.cuda.synchronize()
            assert out.tolist()[1:] == want[1:]
            assert g.census(options=opts) == want       # makes the lists; the captured launches stay as they were
