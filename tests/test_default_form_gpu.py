"""A census with no options anywhere takes the library's form of choice; a form that is asked for
runs as asked.  Both give the union walk's counts.  Whole numbers: no tolerance."""
import numpy as np
import pytest
import torch

import graphgen
import paper_1209_6308_gb300 as tc

pytestmark = pytest.mark.gpu

GRAPHS = {"empty": (7, [], []), "one_vertex": (1, [0], [0]), "loops": (4, [1, 2, 1], [1, 2, 1]), "pair": (3, [0, 1], [1, 0]),
          "star": (500, [0] * 499, list(range(1, 500))), "gnp": graphgen.gnp(130, 0.3, 5), "rmat": graphgen.rmat(12, 16, 0.2, 3),
          "chung_lu": graphgen.chung_lu(9_001, 8.0, 2.1, 0.1, 4, 2)}


@pytest.mark.parametrize("name", GRAPHS)
def test_no_options_give_the_union_walks_counts(name):
    n, s, d = GRAPHS[name]
    s, d = np.asarray(s, np.uint32), np.asarray(d, np.uint32)
    with tc.Graph.from_arcs(n, s, d) as g, tc.Graph.from_arcs(n, s, d, options={"algo": tc.TC_ALGO_UNION}) as u:
        want = u.census()
        assert g.census() == want
        assert g.census(options={"algo": tc.TC_ALGO_UNION}) == want
        out = torch.zeros(16, dtype=torch.int64, device="cuda")
        tc.tc_census_async(g.handle, out)
        assert out.cpu().tolist()[1:] == want[1:]
        with tc.Stream(n, 10) as stream:
            stream.push(s, d, np.zeros(len(s), np.uint64))
            assert stream.census(0)[0] == want


@pytest.mark.parametrize("census_first", [False, True])
def test_captured_without_options(census_first):
    """The captured call takes the form that has a plan: the library's after a census, else the one that
    the same options planned."""
    n, s, d = GRAPHS["rmat"]
    with tc.Graph.from_arcs(n, s, d) as g, tc.Graph.from_arcs(n, s, d, options={"algo": tc.TC_ALGO_UNION}) as u:
        want = u.census()
        if census_first:
            assert g.census() == want
        else:
            tc.tc_census_shard_bounds(g.handle, 1)
        out = torch.zeros(16, dtype=torch.int64, device="cuda")
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            tc.tc_census_async(g.handle, out, stream=torch.cuda.current_stream().cuda_stream)
        graph.replay()
        torch.cuda.synchronize()
        assert out.tolist()[1:] == want[1:]
        assert g.census() == want
