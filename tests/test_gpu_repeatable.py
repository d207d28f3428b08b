"""Queries crowded along boundary edges: a query's bits do not depend on its neighbours.

Each such query has ill-conditioned terms, which a warp evaluates in FP64 from a queue of
its own; 20,000 queries within 1e-3 edge lengths of a short boundary's edges put more on
it than it holds.  A repeated call, a permuted one and the allocation-free entry point
must give the same bits, however the warps are composed.
"""
import ctypes

import numpy as np
import pytest

import gen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def rim(rng):
    """One loop of 200 edges (summed edge by edge)."""
    t = 2 * np.pi * np.arange(200) / 200
    V = np.concatenate([np.stack([np.cos(t), np.sin(t), 0.1 * np.cos(5 * t)], 1), [[0, 0, 0.3]]])
    i = np.arange(200)
    return V, np.stack([np.full(200, 200), i, (i + 1) % 200], 1)


def triangles(rng):
    """100 triangle loops."""
    m = gen.random_soup(100, rng)
    return m.V, m.F


def stacked_quads(rng, copies=4):
    """Unwelded copies of each of 400 small quads: the hierarchy, with several copies of an edge in a leaf."""
    c = rng.random((400, 1, 3))
    u = 0.02 * rng.standard_normal((400, 2, 3))
    quad = np.concatenate([c, c + u[:, :1], c + u[:, :1] + u[:, 1:], c + u[:, 1:]], 1)
    V = np.repeat(quad, copies, 0).reshape(-1, 3)
    b = 4 * np.arange(400 * copies)[:, None]
    return V, np.concatenate([b + [0, 1, 2], b + [0, 2, 3]])


def taller_stacks(rng):
    return stacked_quads(rng, 6)


@pytest.mark.parametrize("kind,n", [("rim", 3_000), ("rim", 20_000), ("triangles", 6_000), ("triangles", 20_000), ("stacked_quads", 60_000),
                                    ("taller_stacks", 60_000)])
def test_same_bits_along_edges(kind, n):
    import paper_2605_01536_gb300 as gwn
    rng = np.random.default_rng(n)
    V, F = globals()[kind](rng)
    V, F = V.astype(np.float32), F.astype(np.int32)
    E = oracle.boundary(F, len(V))
    e = E[np.sort(rng.integers(0, len(E), n))]
    a, b = V[e[:, 0]].astype(np.float64), V[e[:, 1]].astype(np.float64)
    d = rng.normal(size=a.shape)
    d *= 10.0 ** rng.uniform(-5, -3, (n, 1)) * np.linalg.norm(b - a, axis=1, keepdims=True) / np.linalg.norm(d, axis=1, keepdims=True)
    Q = (a + rng.uniform(0.2, 0.8, (n, 1)) * (b - a) + d).astype(np.float32)
    q = torch.from_numpy(Q).cuda()
    config = {"group_test": 1} if n < 16_384 else {}   # keeps a short call off the one-kernel path
    with gwn.Mesh(V, F, config=config) as m:
        lab, w = m.classify(q, want_w=True)
        for _ in range(3):
            lab2, w2 = m.classify(q, want_w=True)
            assert torch.equal(w2, w) and torch.equal(lab2, lab)
            assert torch.equal(m.query(q)[0], m.query(q)[0])
        perm = torch.randperm(n, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
        labp, wp = m.classify(q[perm].contiguous(), want_w=True)
        assert torch.equal(wp, w[perm]) and torch.equal(labp, lab[perm])
        ls, ws = torch.empty_like(lab), torch.empty_like(w)
        rc = gwn.load().gwn_classify_static(m.handle, ctypes.c_void_p(q.data_ptr()), n, ctypes.c_void_p(ls.data_ptr()),
                                            ctypes.c_void_p(ws.data_ptr()),
                                            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        torch.cuda.synchronize()
        assert rc == 0 and torch.equal(ws, w) and torch.equal(ls, lab)
        assert m.counters()["cancel_overflow"] == 0
    sel = rng.choice(n, 500, replace=False)
    ref = oracle.reference(V, F, Q[sel])
    ok = ref["flags"] == 0
    assert np.abs(w.cpu().numpy()[sel].astype(np.float64) - ref["w_antipodal"])[ok].max() <= 1e-5
