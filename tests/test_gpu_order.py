"""The spatial order of large calls: every query answered once, whatever its place.

Results do not depend on the order, so a permuted or repeated batch must give the
same bits, and a call below the ordering threshold the same crossing numbers.
"""
import ctypes

import numpy as np
import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mesh():
    import paper_2605_01536_gb300 as gwn
    m, rng = gen.displaced_soup(5, 8)
    with gwn.Mesh(m.V, m.F) as g:
        yield g, m, rng


# around the threshold and the sizes where the number of cells changes
@pytest.mark.parametrize("n", [16384, 16385, 131_071, 131_072, 1_048_320, 1_048_321, 1_048_576, 2_097_152])
@pytest.mark.parametrize("spread", ["uniform", "one point", "far outside"])
def test_every_query_is_answered(mesh, n, spread):
    import paper_2605_01536_gb300 as gwn
    g, m, rng = mesh
    k = 4096
    base = gen.queries_uniform_bbox(m.V, k, rng)
    if spread == "one point":
        base[:] = base[0]
    elif spread == "far outside":
        base *= np.float32(50)
    ref_chi = g.chi(torch.from_numpy(base).cuda())
    idx = torch.arange(n, device="cuda") * 1_000_003 % k
    q = torch.from_numpy(base).cuda()[idx].contiguous()
    w, chi = g.query(q)
    assert torch.equal(chi, ref_chi[idx])
    first = torch.full((k,), float("nan"), device="cuda")
    first[idx] = w
    assert torch.equal(first[idx], w)            # equal queries, equal bits
    lab, wc = g.classify(q, want_w=True)
    ls, ws = torch.empty_like(lab), torch.empty_like(wc)
    rc = gwn.load().gwn_classify_static(g.handle, ctypes.c_void_p(q.data_ptr()), n, ctypes.c_void_p(ls.data_ptr()),
                                        ctypes.c_void_p(ws.data_ptr()),
                                        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0 and torch.equal(ls, lab)
    assert torch.max(torch.abs(ws - wc)).item() <= 1e-5
