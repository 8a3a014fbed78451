"""Tiles of the scan and of the sort that stop waiting for their predecessors sum these predecessors' input
themselves.  In the library a tile waits long enough never to do so; here it is built to look once, and
the structure and the counts must be the same.  Whole numbers: no tolerance."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_1209_6308_gb300 import _build

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def impatient(tmp_path_factory):
    """libtc.so with primitives.cu compiled for one look."""
    out = tmp_path_factory.mktemp("impatient")
    objs = []
    for src in _build._sources():
        name = os.path.basename(src)
        obj = os.path.join(_build.OBJ, name + ".o")
        if name == "primitives.cu" or not os.path.exists(obj):
            obj = str(out / (name + ".o"))
            extra = ["-DTC_LOOKS=1"] if name == "primitives.cu" else []
            subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, *extra, "-c", src, "-o", obj], check=True)
        objs.append(obj)
    lib = str(out / "libtc.so")
    subprocess.run([_build.nvcc(), *_build.ARCH, "-shared", "-o", lib, *objs, "-cudart", "static"], check=True)
    return lib


def check(lib):
    """In a process of its own: builds, 64 states and scans over many tiles, as the ordinary library's tests
    make them."""
    import graphgen
    import oracle
    import paper_1209_6308_gb300 as tc
    from test_build_gpu import reference
    tc.LIB_PATH = lib
    for n, m in ((2, 3), (4097, 6145), (70_000, 300_001), (262_145, 2_000_003)):
        rng = np.random.default_rng(n)
        s, d = (rng.integers(0, n, m).astype(np.uint32) for _ in range(2))
        off, adj, new, loops, dups = reference(n, s.astype(np.int64), d.astype(np.int64))
        for _ in range(3):
            with tc.Graph.from_arcs(n, s, d) as g:
                o, a, p = tc.tc_graph_export_csr(g.handle)
                assert (p == new).all() and (o == off).all() and (a == adj).all()
    n, s, d = graphgen.rmat(13, 16, 0.2, 5)
    with tc.Graph.from_arcs(n, s, d) as g:
        assert g.census() == oracle.census_bm(n, s, d)
        assert g.census64() == oracle.census64(n, s, d)
    print("same")


def test_tiles_that_give_up(impatient):
    code = f"import sys; sys.path[:0] = [{os.path.dirname(HERE)!r}, {HERE!r}]; import test_lookback_gpu as t; t.check({impatient!r})"
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("same"), r.stdout + r.stderr
