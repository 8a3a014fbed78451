"""A sharded census with no options anywhere takes the form that the whole census takes."""
import numpy as np
import pytest
import torch

import graphgen
import paper_1209_6308_gb300 as tc

pytestmark = pytest.mark.gpu


def _shards(g, world):
    out = torch.zeros(16, dtype=torch.int64, device="cuda")
    total = np.zeros(16, np.int64)
    for r in range(world):
        tc.tc_census_shard(g.handle, out, r, world)
        total += out.cpu().numpy()
    return total.tolist()


@pytest.mark.parametrize("world", [1, 3])
def test_shards_take_the_form_of_the_whole_census(world):
    """The shards' bounds are those of the triangle form's plan, which is cut by other work than the union
    walk's; a graph made with options keeps the form these name."""
    n, s, d = graphgen.rmat(13, 16, 0.2, 5)
    bounds = {}
    for algo in (tc.TC_ALGO_UNION, tc.TC_ALGO_TRIANGLE):
        with tc.Graph.from_arcs(n, s, d, options={"algo": algo}) as g:
            bounds[algo] = tc.tc_census_shard_bounds(g.handle, world)
            want = g.census()
    assert (bounds[tc.TC_ALGO_UNION] != bounds[tc.TC_ALGO_TRIANGLE]).any()
    with tc.Graph.from_arcs(n, s, d) as g:
        assert (tc.tc_census_shard_bounds(g.handle, world) == bounds[tc.TC_ALGO_TRIANGLE]).all()
        assert (tc.tc_census_shard_bounds(g.handle, world, options={}) == bounds[tc.TC_ALGO_UNION]).all()
        assert _shards(g, world)[1:] == want[1:]


@pytest.mark.parametrize("first", ["nothing else", "a census", "a 64-state census"])
def test_captured_shard_takes_the_plan_that_has_its_shards(first):
    """Captured without options: the shards were planned by a call whose algo is 0, and the whole census's
    form may have a plan without shards."""
    n, s, d = graphgen.rmat(12, 16, 0.2, 3)
    with tc.Graph.from_arcs(n, s, d) as g:
        want = g.census(options={"algo": tc.TC_ALGO_SUFFIX})
        if first == "a census":
            assert g.census() == want
        elif first != "nothing else":
            g.census64()
        tc.tc_census_shard_bounds(g.handle, 1, options={})
        out = torch.zeros(16, dtype=torch.int64, device="cuda")
        capture = torch.cuda.CUDAGraph()
        with torch.cuda.graph(capture):
            tc.tc_census_shard(g.handle, out, 0, 1, stream=torch.cuda.current_stream().cuda_stream)
        capture.replay()
        torch.cuda.synchronize()
        assert out.tolist()[1:] == want[1:]
