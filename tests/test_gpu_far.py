"""The boundary hierarchy (far-field expansions) against the oracle and the direct sum.

Tolerance: an accepted expansion is truncated at 1e-7 and a query takes some
hundreds of them, of random sign; the FP32 terms add their usual rounding.  The
library's bar, 1e-5 off the boundary curve, holds with a wide margin; against the
direct kernel's own rounding the same bar is used.
"""
import ctypes

import numpy as np
import pytest

import gen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5
MIN_ORDERED = 16384   # smaller calls take the direct sum


@pytest.fixture(scope="module")
def gwn():
    import paper_2605_01536_gb300 as g
    g.load()
    return g


def disk(n, wave=0.05):
    """Fan over a wavy rim of n vertices: one loop, which the hierarchy's leaves cut (chords)."""
    t = 2 * np.pi * np.arange(n) / n
    r = 1 + wave * np.sin(40 * t)
    V = np.concatenate([np.stack([r * np.cos(t), r * np.sin(t), wave * np.cos(23 * t)], 1), [[0, 0, 0.3]]])
    i = np.arange(n)
    F = np.stack([np.full(n, n), i, (i + 1) % n], 1)
    return V.astype(np.float32), F.astype(np.int32)


def holes_and_rims(level, seed):
    """Small holes (whole loops in a leaf), a large rim, and loops that straddle leaves."""
    m, rng = gen.displaced_soup(level, seed, hole_p=0.05)
    V, F = disk(1500)
    return (np.concatenate([m.V, 0.4 * V + np.float32([0, 0, 2])]).astype(np.float32),
            np.concatenate([m.F, F + m.nv]).astype(np.int32))


MESHES = {
    "rim5000": lambda: disk(5000),
    "rim2049": lambda: disk(2049, 0.0),
    "mixed": lambda: holes_and_rims(6, 3),
    "soup6": lambda: (lambda m: (m.V, m.F))(gen.displaced_soup(6, 9)[0]),
    "tiny scale": lambda: (lambda m: (m.V * np.float32(2.0 ** -20), m.F))(gen.displaced_soup(6, 9)[0]),
    "large scale": lambda: (lambda m: (m.V * np.float32(2.0 ** 40), m.F))(gen.displaced_soup(6, 9)[0]),
}


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("n", [100_003, 262_144])   # the direct sum's work is above the rule's 5e9 operations
def test_far_matches_oracle_and_direct(gwn, name, n):
    V, F = MESHES[name]()
    rng = np.random.default_rng(1)
    ext = float((V.max(0) - V.min(0)).max())
    Q = np.concatenate([gen.queries_uniform_bbox(V, n // 2, rng), gen.queries_near_surface(V, F, n - n // 2 - 64, rng, 1e-3 * ext),
                        (100 * ext * rng.normal(size=(64, 3))).astype(np.float32)])
    q = torch.from_numpy(Q).cuda()
    with gwn.Mesh(V, F) as m, gwn.Mesh(V, F, config={"queries_per_thread": 4}) as d:
        w, chi = m.query(q)
        wd, chid = d.query(q)
        assert torch.equal(chi, chid)
        assert torch.max(torch.abs(w - wd)).item() <= TOL
        assert not torch.equal(w, wd)   # the hierarchy was taken
        perm = torch.randperm(n, device="cuda")
        wp, _ = m.query(q[perm].contiguous())
        assert torch.equal(wp, w[perm])   # a query's result does not depend on the others
        lab, wc = m.classify(q, want_w=True)
        labs, ws = torch.empty_like(lab), torch.empty_like(wc)
        rc = gwn.load().gwn_classify_static(m.handle, ctypes.c_void_p(q.data_ptr()), n, ctypes.c_void_p(labs.data_ptr()),
                                            ctypes.c_void_p(ws.data_ptr()),
                                            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0 and torch.equal(labs, lab) and torch.max(torch.abs(ws - wc)).item() <= TOL
    sel = np.concatenate([rng.choice(n - 64, 400, replace=False), np.arange(n - 64, n)])
    ref = oracle.reference(V, F, Q[sel])
    ok = ref["flags"] == 0
    assert np.array_equal(chi.cpu().numpy()[sel], ref["chi"])
    assert np.max(np.abs(w.cpu().numpy()[sel].astype(np.float64) - ref["w_antipodal"])[ok]) <= TOL
    assert np.array_equal(lab.cpu().numpy()[sel][ok], (ref["w_antipodal"][ok] > 0.5).astype(np.uint8))


@pytest.mark.parametrize("config", [{"quantize_bits": 30}, {"group_test": 2}])
def test_far_modes(gwn, config):
    m6, rng = gen.displaced_soup(6, 9)
    Q = np.concatenate([gen.queries_uniform_bbox(m6.V, 30_000, rng), gen.queries_near_surface(m6.V, m6.F, 30_000, rng)])
    q = torch.from_numpy(Q).cuda()
    with gwn.Mesh(m6.V, m6.F, config=config) as m, gwn.Mesh(m6.V, m6.F, config={**config, "queries_per_thread": 4}) as d:
        w, chi = m.query(q)
        wd, chid = d.query(q)
    assert torch.equal(chi, chid) and torch.max(torch.abs(w - wd)).item() <= TOL


def test_far_queries_at_the_boundary(gwn):
    """Queries 1e-6 to 3e-5 edge lengths off boundary edges, and straight below boundary vertices."""
    V, F = MESHES["mixed"]()
    E = oracle.boundary(F, len(V))
    rng = np.random.default_rng(2)
    e = rng.integers(0, len(E), 65_536)
    a, b = V[E[e, 0]].astype(np.float64), V[E[e, 1]].astype(np.float64)
    t = rng.uniform(0.2, 0.8, (len(e), 1))
    off = rng.normal(size=a.shape)
    d = 10.0 ** rng.uniform(-6, -4.5, (len(e), 1)) * np.linalg.norm(b - a, axis=1, keepdims=True)
    Q = (a + t * (b - a) + d * off / np.linalg.norm(off, axis=1, keepdims=True)).astype(np.float32)
    Q[::4] = V[E[e[::4], 0]] - np.float32([0, 0, 0.5])
    q = torch.from_numpy(Q).cuda()
    with gwn.Mesh(V, F) as m:
        w, chi = m.query(q)
    sel = rng.choice(len(Q), 600, replace=False)
    ref = oracle.reference(V, F, Q[sel])
    ok = ref["flags"] == 0
    assert np.array_equal(chi.cpu().numpy()[sel], ref["chi"])
    assert np.max(np.abs(w.cpu().numpy()[sel].astype(np.float64) - ref["w_antipodal"])[ok]) <= TOL


@pytest.mark.parametrize("name", ["rim5000", "mixed", "soup6"])
def test_far_gradient(gwn, name):
    """Algorithm 3's FP32 bound (test_gpu_gradient.py) plus the truncation of the expansions: at most
    2e-6 / box side each, of random sign over some hundreds of them."""
    V, F = MESHES[name]()
    rng = np.random.default_rng(4)
    ext = float((V.max(0) - V.min(0)).max())
    n = 17_001
    Q = np.concatenate([gen.queries_uniform_bbox(V, n // 2, rng), gen.queries_near_surface(V, F, n - n // 2, rng, 1e-3)])
    q = torch.from_numpy(Q).cuda()
    with gwn.Mesh(V, F) as m:
        g = m.gradient(q)
        perm = torch.randperm(n, device="cuda")
        assert torch.equal(m.gradient(q[perm].contiguous()), g[perm])
    sel = rng.choice(n, 500, replace=False)
    ref, a, c, fl = oracle.gradient(V, oracle.boundary(F, len(V)), Q[sel])
    ok = fl == 0
    tol = 2.0 ** -24 * (128.0 * c + 128.0 * a) + 3e-5 / ext
    assert not (ok[:, None] & (np.abs(g.cpu().numpy()[sel].astype(np.float64) - ref) > tol[:, None])).any()
