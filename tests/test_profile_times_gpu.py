"""The per-CTA times of a profiled census in the triangle form: every entry is of a CTA that took part in
the walk from its start."""
import pytest
import torch

import graphgen
import paper_1209_6308_gb300 as tc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale,ctas", [(16, 0), (16, 1), (16, 8), (19, 0)])
def test_every_cta_is_there_from_the_start(scale, ctas):
    """The last CTA starts before the first one ends (each works until the walk runs out of items)."""
    n, s, d = graphgen.rmat(scale, 16, 0.2, 1)
    opts = {"algo": tc.TC_ALGO_TRIANGLE, "ctas_per_sm": ctas}
    grid = tc.tc_census_grid(opts)
    out, vcost = (torch.zeros(k, dtype=torch.int64, device="cuda") for k in (16, n))
    phase = torch.zeros(3 * grid + 3, dtype=torch.int64, device="cuda")
    with tc.Graph.from_arcs(n, s, d) as g:
        want = g.census(options={"algo": tc.TC_ALGO_SUFFIX})
        for _ in range(2):
            tc.tc_census_profile(g.handle, out, vcost, phase, options=opts)
        torch.cuda.synchronize()
    assert out.tolist()[1:] == want[1:]
    times = phase.view(-1, 3).cpu()
    assert (times[-1] == 0).all()                      # nothing past the grid's entries
    start, items, end = times[:-1].unbind(1)
    assert (start > 0).all() and (start <= items).all() and (items <= end).all()
    assert start.max() < end.min()
