"""Triangle loops over the documented coordinate range (magnitudes below 2^60).

Scaling mesh and queries by a power of two changes no exact value, so crossing numbers
and labels must stay and w must agree with the unscaled result.  Tolerance: the
library's 1e-5 between two evaluations, plus what 1e-37 beside the squared distances
changes at the smallest scale (the queries keep 0.2 to every vertex: at most 1e-37 /
(0.2^2 4^-50) = 3e-6 of an angle).
"""
import ctypes

import numpy as np
import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 2e-5


@pytest.mark.parametrize("k", [-50, -45, 44, 50, 58])
@pytest.mark.parametrize("nt", [3, 200])
def test_scaled_by_a_power_of_two(k, nt):
    import paper_2605_01536_gb300 as gwn
    rng = np.random.default_rng(7)
    mesh = gen.random_soup(nt, rng)
    Q = rng.uniform(-0.6, 1.6, (200_000, 3)).astype(np.float32)
    d2 = np.full(len(Q), np.inf)
    for v in mesh.V:
        d2 = np.minimum(d2, ((Q - v) ** 2).sum(1))
    Q = Q[d2 > 0.04][:17_000]
    n = len(Q)
    assert n >= 16_384   # past the small calls and into the spatial order
    got = []
    for s in (1.0, 2.0 ** k):
        q = torch.from_numpy(Q * np.float32(s)).cuda()
        with gwn.Mesh(mesh.V * np.float32(s), mesh.F) as m, gwn.Batch([m], [n]) as b:
            w, chi = m.query(q)
            lab, wc = m.classify(q, want_w=True)
            ls, ws = torch.empty_like(lab), torch.empty_like(wc)
            rc = gwn.load().gwn_classify_static(m.handle, ctypes.c_void_p(q.data_ptr()), n,
                                                ctypes.c_void_p(ls.data_ptr()), ctypes.c_void_p(ws.data_ptr()),
                                                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
            wb, _ = b.run(q)
            torch.cuda.synchronize()
        assert rc == 0
        got.append([x.cpu().numpy() for x in (chi, lab, ls, w, wc, ws, wb)])
    ref, out = got
    clear = np.abs(ref[3] - 0.5) > 2 * TOL
    assert np.array_equal(out[0], ref[0])
    assert np.array_equal(out[1][clear], ref[1][clear]) and np.array_equal(out[2][clear], ref[2][clear])
    for a, b in zip(out[3:], ref[3:]):
        assert np.isfinite(a).all() and np.abs(a.astype(np.float64) - b).max() <= TOL


@pytest.mark.parametrize("k", [-40, -44])
def test_below_vertices_at_small_scales(k):
    """Queries straight below vertices at 1e-4 to 1 edge lengths, down to distances of 1e-18, where 1e-37
    beside the squared distance shortens a unit vector by far more than rounding.  (Beside a vertex the
    edges' own terms are off there; straight below it n and d shrink alike, down to 2^-44.)"""
    import paper_2605_01536_gb300 as gwn
    rng = np.random.default_rng(3)
    mesh = gen.random_soup(400, rng)
    p = mesh.V[rng.integers(0, len(mesh.V), 17_000)]
    Q = (p - np.float32([0, 0, 1]) * (0.2 * 10.0 ** rng.uniform(-4, 0, (len(p), 1)))).astype(np.float32)
    got = []
    for s in (np.float32(1), np.float32(2.0 ** k)):
        q = torch.from_numpy(Q * s).cuda()
        with gwn.Mesh(mesh.V * s, mesh.F) as m, gwn.Batch([m], [len(Q)]) as b:
            got.append([x.cpu().numpy().astype(np.float64) for x in (m.query(q)[0], m.classify(q, want_w=True)[1], b.run(q)[0])])
    for a, b in zip(got[1], got[0]):
        assert np.abs(a - b).max() <= TOL, np.abs(a - b).max()
