"""Calls of more than 2^31 / 3 queries: coordinates beyond the 32-bit range of indices.

A call may have 2^31 - 1 queries.  Queries near the margin are listed for the FP64
re-evaluation; the ones at the end of this call lie beyond float 2^31 of the array and must
get what a call of their own gives them.
"""
import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_listed_queries_beyond_two_to_the_31_floats():
    import paper_2605_01536_gb300 as gwn
    if torch.cuda.mem_get_info()[0] < 80 << 30:
        pytest.skip("needs 80 GB of device memory")
    n, tail = 720_000_000, 4_000_000   # 3 n > 2^31 from query 715,827,883 on
    mesh = gen.small_cap(3, 0.8)
    q = torch.empty((n, 3), dtype=torch.float32, device="cuda")
    q.uniform_(-1.5, 1.5, generator=torch.Generator("cuda").manual_seed(5))
    with gwn.Mesh(mesh.V, mesh.F, config={"classify_margin": 1e-3}) as m:
        lab, w = m.classify(q, want_w=True)
        lab_t, w_t = lab[-tail:].clone(), w[-tail:].clone()
        del lab, w
        m.counters(reset=True)
        lab_s, w_s = m.classify(q[-tail:].contiguous(), want_w=True)
        listed = m.counters()["fp64_reevaluations"]
    assert listed > 100
    assert torch.equal(lab_t, lab_s) and torch.max(torch.abs(w_t - w_s)).item() <= 2e-6
