"""gwn_classify_static cuts large calls into slices that fit its scratch: w and labels are gwn_classify's to the bit."""
import ctypes

import numpy as np
import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def triangles(n, rng):
    V = (rng.random((n, 1, 3)) + 0.1 * rng.standard_normal((n, 3, 3))).reshape(-1, 3).astype(np.float32)
    return V, np.arange(3 * n, dtype=np.int32).reshape(-1, 3)


MESHES = {
    "staircase": lambda rng: (lambda m: (m.V, m.F))(gen.staircase_sphere(20.0)),   # a short boundary in a few parts
    "triangles": lambda rng: triangles(3000, rng),                                 # triangle loops
    "soup": lambda rng: (lambda m: (m.V, m.F))(gen.displaced_soup(6, seed=2)[0]),  # the hierarchy
}


@pytest.mark.parametrize("name,n", [("staircase", 16383), ("staircase", 100000), ("staircase", 524288), ("staircase", 2097152),
                                    ("triangles", 16384), ("triangles", 200000), ("soup", 400000), ("soup", 1048577)])
def test_same_bits(name, n):
    import paper_2605_01536_gb300 as gwn
    rng = np.random.default_rng(n)
    V, F = MESHES[name](rng)
    q = torch.from_numpy(gen.queries_uniform_bbox(V, n, rng)).cuda()
    with gwn.Mesh(V, F) as m:
        label, w = m.classify(q, want_w=True)
        ls, ws = torch.empty_like(label), torch.empty_like(w)
        rc = gwn.load().gwn_classify_static(m.handle, ctypes.c_void_p(q.data_ptr()), n, ctypes.c_void_p(ls.data_ptr()),
                                            ctypes.c_void_p(ws.data_ptr()),
                                            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        torch.cuda.synchronize()
    assert rc == 0 and torch.equal(ls, label) and torch.equal(ws, w)
