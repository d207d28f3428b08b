"""Build of meshes with one vertex of many unmatched edges: the time does not jump with their number."""
import time

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def star(spokes, rng):
    """Triangles that share only vertex 0: two unmatched edges each at it."""
    V = rng.random((1 + 2 * spokes, 3)).astype(np.float32)
    i = 1 + 2 * rng.permutation(spokes)[:, None]
    return V, np.concatenate([np.zeros_like(i), i, i + 1], 1).astype(np.int32)


def best_build(V, F, reps=20):
    import paper_2605_01536_gb300 as gwn
    v, f = torch.from_numpy(V).cuda(), torch.from_numpy(F).cuda()
    best = 1e9
    with gwn.Mesh(V, F) as keep:   # holds the memory pool
        edges = keep.boundary_edges()
        for _ in range(reps):
            m = gwn.Mesh(v, f, build=False)
            torch.cuda.synchronize()
            t = time.perf_counter()
            m.build()
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
            m.close()
    return best, edges


@pytest.mark.parametrize("spokes", [1, 2, 31, 63, 64, 65, 400])
def test_star_edges(spokes):
    V, F = star(spokes, np.random.default_rng(spokes))
    _, edges = best_build(V, F, 1)
    assert np.array_equal(edges, oracle.boundary(F, len(V)))


def test_star_time():
    """63 spokes (126 half-edges at the vertex) against 2: a generous factor over the same launches."""
    few, _ = best_build(*star(2, np.random.default_rng(0)))
    many, _ = best_build(*star(63, np.random.default_rng(1)))
    assert many <= 2.0 * few, (many, few)
