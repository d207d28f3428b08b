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


@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 1), (33, 1, 5), (7, 40, 17), (130, 3, 16), (64, 70, 33)])
def test_grid_rasterisation_on_any_axes(nx, ny, nz):
    """Unsorted axes with repeated entries; triangles from smaller than a cell to the whole grid."""
    import paper_2605_01536_gb300 as gwn
    rng = np.random.default_rng(nx * ny)
    small = gen.random_soup(300, rng)
    V = np.concatenate([small.V, np.float32([[-9, -9, .3], [9, -9, .3], [0, 9, .9], [-1, -1, -1], [2, -1, -1], [-1, 2, 2]])])
    F = np.concatenate([small.F, small.nv + np.array([[0, 1, 2], [3, 4, 5]], np.int32)])
    axis = lambda n: rng.choice(np.linspace(-0.2, 1.2, 2 * n + 1), n).astype(np.float32)
    x, y, z = axis(nx), axis(ny), np.sort(axis(nz))
    Z, Y, X = np.meshgrid(z, y, x, indexing="ij")
    P = torch.from_numpy(np.stack([X, Y, Z], -1).reshape(-1, 3).astype(np.float32)).cuda()
    with gwn.Mesh(V, F) as m:
        assert torch.equal(m.grid_chi(x, y, z).ravel(), m.chi(P))
        lab, w = m.classify_grid(x, y, z, want_w=True)
        ref_lab, ref_w = m.classify(P, want_w=True)
    assert torch.equal(lab.ravel(), ref_lab) and torch.max(torch.abs(w.ravel() - ref_w)).item() <= 1e-5
