"""The built structure (relabelling, offsets, flagged lists) against a numpy restatement, at sizes
around the tiles of the sort (6144 keys) and the scan (4096 values).  Whole numbers: no tolerance."""
import numpy as np
import pytest

import paper_1209_6308_gb300 as tc

pytestmark = pytest.mark.gpu


def reference(n, s, d):
    """(off, adj, new_of_old, loops, dups): Fig. 7's structure in ids of descending degree."""
    keep = s != d
    arcs = np.unique(s[keep].astype(np.int64) * n + d[keep])
    s2, d2 = arcs // n, arcs % n
    lo, hi = np.minimum(s2, d2), np.maximum(s2, d2)
    pair, inv = np.unique(lo * n + hi, return_inverse=True)
    dirs = np.zeros(len(pair), np.int64)
    np.bitwise_or.at(dirs, inv, np.where(s2 < d2, 1, 2))
    lo, hi = pair // n, pair % n
    deg = np.bincount(lo, minlength=n) + np.bincount(hi, minlength=n)
    order = np.lexsort((np.arange(n), -deg))
    new = np.empty(n, np.int64)
    new[order] = np.arange(n)
    own = np.concatenate([new[lo], new[hi]])
    nbr = np.concatenate([new[hi], new[lo]])
    dd = np.concatenate([dirs, (dirs & 1) << 1 | dirs >> 1])
    at = np.lexsort((nbr, own))
    off = np.concatenate([[0], np.cumsum(np.bincount(own, minlength=n))]).astype(np.uint64)
    return off, (nbr[at] << 2 | dd[at]).astype(np.uint32), new.astype(np.uint32), int((~keep).sum()), int(keep.sum() - len(arcs))


@pytest.mark.parametrize("n,m", [(1, 0), (2, 3), (5, 40), (4095, 6143), (4096, 6144), (4097, 6145), (300, 100_000),
                                 (8192, 12_288), (6145, 16_384), (20_001, 65_537), (70_000, 300_001), (262_145, 1_000_003)])
@pytest.mark.parametrize("skew", [False, True])
def test_build_matches_the_reference(n, m, skew):
    rng = np.random.default_rng(n + m)
    s = rng.integers(0, n, m) if not skew else (n * rng.random(m) ** 4).astype(np.int64)
    d = rng.integers(0, n, m)
    s, d = s.astype(np.uint32), d.astype(np.uint32)
    off, adj, new, loops, dups = reference(n, s.astype(np.int64), d.astype(np.int64))
    with tc.Graph.from_arcs(n, s, d) as g:
        o, a, p = tc.tc_graph_export_csr(g.handle)
        st = g.stats()
        np.testing.assert_array_equal(p, new)
        np.testing.assert_array_equal(o, off)
        np.testing.assert_array_equal(a, adj)
        assert (st["loops_dropped"], st["dups_dropped"], st["e_sym"]) == (loops, dups, len(adj) // 2)
        with tc.Graph.from_csr(n, o, a) as h:       # ids already descend by degree: the same structure
            o2, a2, p2 = tc.tc_graph_export_csr(h.handle)
            np.testing.assert_array_equal(o2, off)
            np.testing.assert_array_equal(a2, adj)
            np.testing.assert_array_equal(p2, np.arange(n, dtype=np.uint32))
            if n <= 20_001:
                forms = [h.census(options={"algo": a}) for a in (0, 1, 2)] + [g.census(options={"algo": 2})]
                assert all(f == forms[0] for f in forms)
