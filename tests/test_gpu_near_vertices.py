"""Queries 1e-2 to 1e-6 edge lengths from vertices, against the FP64 oracle.

Seen from beside a vertex the triangle's other two vertices are far away, and a
determinant taken with a far vertex's relative vector loses the distance's share of
its digits.  The library's bar, 1e-5, holds at every distance; labels are exact.
Queries within 1e-6 of the scene's coordinates sit a few units of rounding beside the
vertex, which the oracle sees as well (it takes the same FP32 inputs).
"""
import numpy as np
import pytest

import gen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5


def beside_vertices(V, F, n, rng, lo=-6.0, hi=-2.0):
    """Points at 10^lo to 10^hi times an edge's length from a corner of a random face."""
    f = F[rng.integers(0, len(F), n)]
    c = np.arange(n) % 3
    p = V[f[np.arange(n), c]].astype(np.float64)
    e = np.linalg.norm(V[f[np.arange(n), (c + 1) % 3]] - p, axis=1, keepdims=True)
    d = rng.normal(size=(n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    return (p + 10.0 ** rng.uniform(lo, hi, (n, 1)) * e * d).astype(np.float32)


def slim(nt, rng):
    """Triangles with one edge a thousandth of the others."""
    V = gen.random_soup(nt, rng).V.reshape(-1, 3, 3).copy()
    k = np.arange(nt) % 3
    i = np.arange(nt)
    V[i, (k + 1) % 3] = V[i, k] + 1e-3 * (V[i, (k + 1) % 3] - V[i, k])
    return V.reshape(-1, 3).astype(np.float32), np.arange(3 * nt, dtype=np.int32).reshape(-1, 3)


def soup(nt, rng):
    m = gen.random_soup(nt, rng)
    return m.V, m.F


def one_face_holes(nt, rng):
    """A scan with one-face holes: a sphere with every ninth face left out."""
    V, F = sphere()
    return V, F[np.arange(len(F)) % 9 != 0]


def sphere():
    V, F = gen.icosphere(4)
    return V.astype(np.float32), F.astype(np.int32)


LOOPS = {"soup": soup, "slim": slim, "holes": one_face_holes}


@pytest.mark.parametrize("kind", list(LOOPS))
@pytest.mark.parametrize("n", [6_000, 17_000])
def test_triangle_loops_beside_vertices(kind, n):
    import paper_2605_01536_gb300 as gwn
    rng = np.random.default_rng(n)
    V, F = LOOPS[kind](600, rng)
    Q = beside_vertices(V, F, n, rng)
    sel = rng.choice(n, 3_000, replace=False)
    ref = oracle.reference(V, F, Q[sel])
    ok = ref["flags"] == 0
    q = torch.from_numpy(Q).cuda()
    with gwn.Mesh(V, F) as m, gwn.Batch([m], [n]) as b:
        w, chi = m.query(q)
        lab, wc = m.classify(q, want_w=True)
        wb, _ = b.run(q)
        torch.cuda.synchronize()
    assert np.array_equal(chi.cpu().numpy()[sel], ref["chi"])
    for x in (w, wc, wb):
        err = np.abs(x.cpu().numpy()[sel].astype(np.float64) - ref["w_antipodal"])[ok]
        assert err.max() <= TOL, err.max()
    assert np.array_equal(lab.cpu().numpy()[sel][ok], (ref["w_antipodal"][ok] > 0.5).astype(np.uint8))


DIRECT = {
    "soup": lambda rng: soup(300, rng),
    "slim": lambda rng: slim(300, rng),
    "cap": lambda rng: (lambda m: (m.V, m.F))(gen.small_cap(4, 0.8)),
    "closed": lambda rng: sphere(),
}


@pytest.mark.parametrize("kind", list(DIRECT))
def test_direct_beside_vertices(kind):
    """Queries close to a face's plane, compared with the distance to its vertices, are left out: the
    solid angle jumps inside the face."""
    import paper_2605_01536_gb300 as gwn
    rng = np.random.default_rng(3)
    V, F = DIRECT[kind](rng)
    Q = beside_vertices(V, F, 4_000, rng)
    A, B, C = (V[F[:, i]].astype(np.float64) for i in range(3))
    N = np.cross(B - A, C - A)
    keep = np.ones(len(Q), bool)
    for i, p in enumerate(Q.astype(np.float64)):
        d = np.abs(np.einsum("ij,ij->i", p - A, N)) / np.linalg.norm(N, axis=1)
        e = np.linalg.norm(np.stack([p - A, p - B, p - C]), axis=2).min(0)
        keep[i] = (d > np.minimum(0.03 * e, 1e-4)).all() and e.min() > 0   # (on a vertex w is undefined)
    Q = Q[keep]
    assert len(Q) >= 500
    ref = oracle.direct(V, F, Q)
    with gwn.Mesh(V, F, build=False) as m:
        w = m.direct(torch.from_numpy(Q).cuda()).cpu().numpy().astype(np.float64)
    assert np.abs(w - ref).max() <= TOL, np.abs(w - ref).max()


@pytest.mark.parametrize("k", [-45, 30, 44, 58])
def test_direct_scaled_by_a_power_of_two(k):
    import paper_2605_01536_gb300 as gwn
    rng = np.random.default_rng(5)
    mesh = gen.random_soup(300, rng)
    Q = rng.uniform(-0.6, 1.6, (2_000, 3)).astype(np.float32)
    got = []
    for s in (np.float32(1), np.float32(2.0 ** k)):
        with gwn.Mesh(mesh.V * s, mesh.F, build=False) as m:
            got.append(m.direct(torch.from_numpy(Q * s).cuda()).cpu().numpy().astype(np.float64))
    assert np.abs(got[1] - got[0]).max() <= TOL
