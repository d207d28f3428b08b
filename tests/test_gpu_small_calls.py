"""Calls small enough for one kernel, at its limits, against the oracle (w within 1e-5, chi and labels exact)."""
import ctypes

import numpy as np
import pytest

import gen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def big_fan(n):
    t = 2 * np.pi * np.arange(n) / n
    V = np.concatenate([np.stack([np.cos(t), np.sin(t), 0.2 * np.sin(3 * t)], 1), [[0, 0, 0.3]]])
    return V.astype(np.float32), np.stack([0 * np.arange(n) + n, np.arange(n), (np.arange(n) + 1) % n], 1).astype(np.int32)


MESHES = {
    "one triangle": lambda: (np.eye(3, dtype=np.float32), np.array([[0, 1, 2]], np.int32)),
    "cap": lambda: (lambda m: (m.V, m.F))(gen.small_cap(3, 0.8)),
    "closed": lambda: tuple(a.astype(t) for a, t in zip(gen.icosphere(3), (np.float32, np.int32))),
    "2048 triangles": lambda: big_fan(2048),       # every leaf tested
    "2049 triangles": lambda: big_fan(2049),       # the tree walked
    "4095 points": lambda: big_fan(4094),
    "4097 points": lambda: big_fan(4096),          # the general path
    "staircase": lambda: (lambda m: (m.V, m.F))(gen.staircase_sphere(6.0)),
}


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("n", [1, 33, 257, 4096, 4097])
def test_small_calls(name, n):
    import paper_2605_01536_gb300 as gwn
    V, F = MESHES[name]()
    rng = np.random.default_rng(n)
    Q = np.concatenate([gen.queries_uniform_bbox(V, n - n // 2, rng), gen.queries_near_surface(V, F, n // 2, rng, 1e-4)])
    if n > 200:   # degenerate: on vertices and edge midpoints, below them, and close to edges
        Q[:40] = V[rng.integers(0, len(V), 40)]
        Q[40:80] = 0.5 * (V[F[:, 0]] + V[F[:, 1]])[rng.integers(0, len(F), 40)]
        Q[80:120] = V[rng.integers(0, len(V), 40)] - np.float32([0, 0, 0.25])
        if len(F) >= 40:
            Q[120:160] = gen.queries_near_triangle_edges(V, F, 40, rng)
    sel = np.arange(n) if n <= 300 else np.concatenate([np.arange(160), rng.choice(n, 300, replace=False)])
    ref = oracle.reference(V, F, Q[sel])
    ok = ref["flags"] == 0
    q = torch.from_numpy(Q).cuda()
    with gwn.Mesh(V, F) as m:
        w, chi = m.query(q)
        lab, wc = m.classify(q, want_w=True)
        only = m.classify(q)
        ls, ws = torch.empty_like(lab), torch.empty_like(wc)
        rc = gwn.load().gwn_classify_static(m.handle, ctypes.c_void_p(q.data_ptr()), n, ctypes.c_void_p(ls.data_ptr()),
                                            ctypes.c_void_p(ws.data_ptr()),
                                            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0 and torch.equal(ls, lab) and torch.equal(only, lab)
    assert torch.nan_to_num((ws - wc).abs()).max().item() <= 1e-5
    assert np.array_equal(chi.cpu().numpy()[sel], ref["chi"])
    for x in (w, wc):
        assert np.max(np.abs(x.cpu().numpy()[sel].astype(np.float64) - ref["w_antipodal"])[ok], initial=0) <= 1e-5
    assert np.array_equal(lab.cpu().numpy()[sel][ok], (ref["w_antipodal"][ok] > 0.5).astype(np.uint8))
