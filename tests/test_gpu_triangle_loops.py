"""Boundary loops of three edges summed as one triangle term, against the oracle.

The bar is the library's: crossing numbers bit-exact, w within 1e-5 off the boundary
curve, labels exact.  (A triangle term's rounding is a few units of its own angle;
near a triangle the edge-by-edge terms of the general path decide.)
"""
import numpy as np
import pytest

import gen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module")
def gwn():
    import paper_2605_01536_gb300 as g
    g.load()
    return g


def _mixed(nt, seed):
    """nt random triangles, some degenerate or vertical, and an open cap with a longer loop."""
    rng = np.random.default_rng(seed)
    m = gen.random_soup(nt, rng)
    V = m.V.copy().reshape(-1, 3, 3)
    V[0, 2] = V[0, 1]                                 # zero area
    if nt > 3:
        V[1, 2] = (V[1, 0] + V[1, 1]) / 2             # collinear
        V[2, 1:, 0] = V[2, 0, 0]                      # vertical plane
        V[3] = np.float32([[0, 0, .5], [1, 0, .5], [0, 1, .5]])   # axis-aligned, grid-exact
    cap = gen.small_cap(1, 0.5)
    return (np.concatenate([V.reshape(-1, 3), cap.V + np.float32(2)]).astype(np.float32),
            np.concatenate([m.F, cap.F + 3 * nt]).astype(np.int32), rng)


@pytest.mark.parametrize("nt", [1, 7, 102, 103, 511, 2000])
@pytest.mark.parametrize("n", [1, 700, 16_500])
def test_triangle_loops(gwn, nt, n):
    V, F, rng = _mixed(nt, nt)
    Q = np.concatenate([gen.queries_uniform_bbox(V, n - n // 2, rng), gen.queries_near_surface(V, F, n // 2, rng, 1e-5)])
    if n > 100 and nt > 3:
        k = 64
        Q[:k] = np.concatenate([rng.integers(0, 5, (k, 2)) / 4.0, rng.integers(0, 3, (k, 1)) / 4.0], 1)   # rays through the edges
        Q[k:2 * k] = gen.queries_near_triangle_edges(V, F[4:4 + max(nt - 4, 1)], min(k, max(nt - 4, 1)), rng)[
            rng.integers(0, min(k, max(nt - 4, 1)), k)]
        Q[2 * k:2 * k + 8] = V[rng.integers(0, len(V), 8)]
    q = torch.from_numpy(Q).cuda()
    sel = np.arange(n) if n <= 700 else np.concatenate([np.arange(200), rng.choice(n, 400, replace=False)])
    ref = oracle.reference(V, F, Q[sel])
    ok = ref["flags"] == 0
    with gwn.Mesh(V, F) as m, gwn.Batch([m, m], [n, n]) as b:
        w, chi = m.query(q)
        lab = m.classify(q)
        wb, chib = b.run(torch.cat([q, q]).contiguous())
    for x in (w, wb[:n], wb[n:]):
        assert np.max(np.abs(x.cpu().numpy()[sel].astype(np.float64) - ref["w_antipodal"])[ok], initial=0) <= TOL
    assert np.array_equal(chi.cpu().numpy()[sel], ref["chi"]) and torch.equal(chib[:n], chi)
    assert np.array_equal(lab.cpu().numpy()[sel][ok], (ref["w_antipodal"][ok] > 0.5).astype(np.uint8))
