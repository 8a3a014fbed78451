"""The byte counts the benchmark's rooflines divide by, against a count over the exported lists."""
import numpy as np
import pytest
import torch

import bench
import graphgen
import paper_1209_6308_gb300 as tc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["rmat18", "gnp", "hubs"])
def test_entries_read_as_16_bit_ids(name):
    """Every entry below b of a pair (b, c), b below both 2^17 and the count of vertices of degree above 256,
    and no other one; an entry so read counts 2 B in the triangle form's roofline instead of 4."""
    n, s, d = {"rmat18": lambda: graphgen.rmat(18, 16, 0.2, 3), "gnp": lambda: graphgen.gnp(1500, 0.4, 2),
               "hubs": lambda: graphgen.rmat(13, 64, 0.2, 4)}[name]()
    with tc.Graph.from_arcs(n, s, d) as g:
        off, adj, _ = tc.tc_graph_export_csr(g.handle)
        info = g.stats()
        got = bench.entries_in_16_bits(tc, torch, g)
    deg = np.diff(off.astype(np.int64))
    limit = min(1 << 17, int((deg > 256).sum()))
    owner = np.repeat(np.arange(n), deg)
    position = np.arange(len(adj)) - np.repeat(off[:-1].astype(np.int64), deg)
    b = (adj >> 2).astype(np.int64)
    lower = b < owner                     # b = N[c][p], a pair (b, c) whose walk reads p entries
    assert int(position[lower].sum()) == info["sum_tri_walk"]
    assert got == int(position[lower & (b < limit)].sum()) > 0
    whole = bench.form_roofline(tc, n, info, tc.TC_ALGO_TRIANGLE, 1.0)["bytes_alg_per_launch"]
    assert bench.form_roofline(tc, n, info, tc.TC_ALGO_TRIANGLE, 1.0, got)["bytes_alg_per_launch"] == whole - 2 * got


@pytest.mark.parametrize("name,launches", [("small", 3), ("items", 4), ("dense", 4)])
def test_launches_of_a_census(name, launches):
    """One walk, a walk whose 2^15 items and more have a launch of their own, and the 16-bit walk without a
    vertex past its table's first id."""
    def random(n, degree):
        rng = np.random.default_rng(n)
        return n, *(rng.integers(0, n, n * degree // 2).astype(np.uint32) for _ in range(2))

    n, s, d = {"small": lambda: random(1 << 12, 32), "items": lambda: random(60_000, 100),
               "dense": lambda: graphgen.gnp(2400, 0.5, seed=2400)}[name]()
    with tc.Graph.from_arcs(n, s, d) as g:
        info = g.stats()
        assert (bench.triangle_kernel(info) == "k_walk16") == (name == "dense")
        assert bench.census_launches(tc, g.handle, n, info, tc.TC_ALGO_TRIANGLE) == launches
        assert bench.census_launches(tc, g.handle, n, info, tc.TC_ALGO_SUFFIX) == 1
