"""The matrix census's two routes (sums sampled at the ones of the sparse dyad matrices; whole
products on the tensor cores for dense graphs) around their dispatch line and the product's tile,
depth and pipeline edges.  Counts are whole numbers: no tolerance."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_1209_6308_gb300 as tc

pytestmark = pytest.mark.gpu


# 128 x 256 tiles, 128 columns per stage, 4 stages; whole products from 24 e > n^2 (p about 0.043)
@pytest.mark.parametrize("n", [127, 128, 129, 255, 257, 513, 641, 1025])
@pytest.mark.parametrize("p", [0.02, 0.07, 0.5])
def test_both_routes_match_the_oracle(n, p):
    n, s, d = graphgen.gnp(n, p, seed=7 * n)
    with tc.Graph.from_arcs(n, s, d) as g:
        assert g.census_matrix() == oracle.census_bm(n, s, d)


@pytest.mark.parametrize("n,recip", [(16_383, 0.0), (16_384, 0.5)])
def test_largest_sizes_agree_with_the_census(n, recip):
    _, s, d = graphgen.chung_lu(n, 24.0, 2.1, recip, 9, 2)
    with tc.Graph.from_arcs(n, s, d) as g:
        assert g.census_matrix() == g.census(options={"algo": tc.TC_ALGO_TRIANGLE})


def test_largest_dense_graph_agrees_with_the_census():
    n = 16_384
    rng = np.random.default_rng(3)
    s, d = rng.integers(0, n, (2, n * n // 12)).astype(np.uint32)     # a tenth of the pairs linked or more
    with tc.Graph.from_arcs(n, s, d) as g:
        assert 24 * g.stats()["e_sym"] > n * n
        assert g.census_matrix() == g.census(options={"algo": tc.TC_ALGO_TRIANGLE})
