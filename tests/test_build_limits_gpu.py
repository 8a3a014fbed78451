"""The largest number of connected pairs a graph may have (include/tc.h: below 2^31)."""
import pytest

import paper_1209_6308_gb300 as tc

pytestmark = pytest.mark.gpu


def test_too_many_pairs_are_refused():
    """2^31 arcs a -> 2^16 + b, a < 2^16, b < 2^15, each a pair of its own: TC_ERR_RANGE, and the library
    goes on working."""
    import torch
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 150 << 30:
        pytest.skip("needs about 100 GiB for the arcs and their keys")
    a = torch.arange(1 << 16, device="cuda", dtype=torch.int32).repeat_interleave(1 << 15)
    b = torch.arange(1 << 15, device="cuda", dtype=torch.int32).add_(1 << 16).repeat(1 << 16)
    with pytest.raises(tc.TcError) as e:
        tc.Graph.from_arcs(3 << 15, a, b)
    assert e.value.status == tc.TC_ERR_RANGE and "pairs" in str(e.value)
    with tc.Graph.from_arcs(3 << 15, a[:1000].clone(), b[:1000].clone()) as g:
        assert g.stats()["e_sym"] == 1000
    del a, b
    torch.cuda.empty_cache()
