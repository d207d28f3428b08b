"""Boundary extraction and chaining at the edges of their paths: bit-exact against the oracle."""
import numpy as np
import pytest

import gen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def fan(n, centre_first):
    """n triangles around a centre: a vertex of n + 1 edges and a loop of n."""
    t = 2 * np.pi * np.arange(n) / n
    rim = np.stack([np.cos(t), np.sin(t), 0.1 * np.sin(7 * t)], 1)
    i = np.arange(n)
    if centre_first:   # every edge of the centre falls into its bucket
        return np.concatenate([[[0, 0, 0.2]], rim]), np.stack([0 * i, i + 1, (i + 1) % n + 1], 1)
    return np.concatenate([rim, [[0, 0, 0.2]]]), np.stack([0 * i + n, i, (i + 1) % n], 1)


def repeated():
    """Duplicate, reversed and degenerate faces: net multiplicities 3, 0, -2 and zero chains."""
    V = np.random.default_rng(0).random((9, 3))
    F = [[0, 1, 2]] * 3 + [[3, 4, 5], [5, 4, 3]] + [[6, 8, 7]] * 2 + [[1, 1, 4], [2, 2, 2]]
    return V, np.array(F)


CASES = {f"fan{n}{'c' if c else ''}": (lambda n=n, c=c: fan(n, c))
         for n, c in [(3, True), (47, True), (48, False), (49, True), (127, True), (128, True), (129, True), (16385, False), (40_000, True)]}
CASES["repeated"] = repeated
CASES["soup"] = lambda: (lambda m: (m.V, m.F))(gen.random_soup(5000, np.random.default_rng(1)))
CASES["holes"] = lambda: (lambda m: (m.V, m.F))(gen.displaced_soup(5, 2, hole_p=0.3)[0])


@pytest.mark.parametrize("name", list(CASES))
def test_boundary(name):
    import paper_2605_01536_gb300 as gwn
    V, F = CASES[name]()
    V, F = V.astype(np.float32), F.astype(np.int32)
    E = oracle.boundary(F, len(V))
    with gwn.Mesh(V, F) as m:
        assert np.array_equal(m.boundary_edges(), E)
        P = m.boundary_points()
        q = torch.rand((500, 3), device="cuda") * 2 - 1
        w, chi = m.query(q)
    # the chained points give every edge once, as closed loops
    key = lambda a: np.sort(a.view([("", a.dtype)] * a.shape[1]).ravel())
    a = np.flatnonzero(P[:, 3] != 0)
    got = np.ascontiguousarray(np.concatenate([P[a, :3], P[a + 1, :3]], 1))
    want = np.ascontiguousarray(np.concatenate([V[E[:, 0]], V[E[:, 1]]], 1))
    assert np.array_equal(key(got), key(want))
    ref = oracle.reference(V, F, q.cpu().numpy())
    ok = ref["flags"] == 0
    assert np.array_equal(chi.cpu().numpy(), ref["chi"])
    assert np.max(np.abs(w.cpu().numpy() - ref["w_antipodal"])[ok], initial=0) <= 1e-5
