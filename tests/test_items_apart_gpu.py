"""The general triangle walk of a graph with many CTA items, whose items and one-warp vertices are two
launches.  Counts are whole numbers: no tolerance."""
import numpy as np
import pytest
import torch

import paper_1209_6308_gb300 as tc

pytestmark = pytest.mark.gpu

TRI = {"algo": tc.TC_ALGO_TRIANGLE}


def random(n, degree):
    gen = torch.Generator("cuda").manual_seed(n + degree)
    s, d = (torch.randint(0, n, (n * degree // 2,), device="cuda", generator=gen, dtype=torch.int32) for _ in range(2))
    return n, s, d


def median_ms(call, reps=15):
    times = []
    for _ in range(reps):
        e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        e0.record()
        call()
        e1.record()
        e1.synchronize()
        times.append(e0.elapsed_time(e1))
    return sorted(times)[reps // 2]


# every vertex (all but a few) is one item: 2^15 items lie between the first two
@pytest.mark.parametrize("n", [32_000, 33_500, 60_000])
@pytest.mark.parametrize("warp_max", [64, 100])
def test_counts_and_times_about_the_limit(n, warp_max):
    opts = {**TRI, "warp_max_deg": warp_max}
    grid = tc.tc_census_grid(opts)
    out, vcost = (torch.zeros(k, dtype=torch.int64, device="cuda") for k in (16, n))
    phase = torch.zeros(3 * grid + 3, dtype=torch.int64, device="cuda")
    with tc.Graph.from_arcs(*random(n, 100)) as g:
        want = g.census(options={"algo": tc.TC_ALGO_SUFFIX})
        assert g.census(options=opts) == want
        (i0, v0), (items, v_end) = tc.tc_census_shard_bounds(g.handle, 1, options=opts)
        assert warp_max != 64 or (items - i0 >= 1 << 15) == (n > 32_768)
        total = np.zeros(16, np.int64)
        for r in range(3):
            tc.tc_census_shard(g.handle, out, r, 3, options=opts)
            total += out.cpu().numpy()
        assert total.tolist()[1:] == want[1:]
        tc.tc_census_profile(g.handle, out, vcost, phase, options=opts)
        torch.cuda.synchronize()
    assert out.tolist()[1:] == want[1:]
    times = phase.view(-1, 3).cpu()
    assert (times[-1] == 0).all()
    start, done, end = times[:-1].unbind(1)
    assert (start > 0).all() and (start <= done).all() and (done <= end).all()


def test_many_items_run_at_eight_ctas():
    """2^18 items of about a hundred short lists wait for their loads, so eight CTAs per SM are faster than
    six; were six all that is resident, both options would take the same time."""
    out = torch.zeros(16, dtype=torch.int64, device="cuda")
    with tc.Graph.from_arcs(*random(1 << 18, 100)) as g:
        ms = {}
        for ctas in (6, 8, 6, 8):
            opts = {**TRI, "ctas_per_sm": ctas}
            tc.tc_census_async(g.handle, out, options=opts)
            ms[ctas] = min(ms.get(ctas, float("inf")), median_ms(lambda: tc.tc_census_async(g.handle, out, options=opts)))
    assert ms[8] <= 0.95 * ms[6], ms
