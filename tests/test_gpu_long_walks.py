"""Walks through thousands of nodes, cut (calls of up to 32768 queries) and whole: chi and
the counts of exact decisions are the same however the queries are split, chi the oracle's."""
import numpy as np
import pytest

import gen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def rough_field(k, rng):
    """k x k integer-lattice height field on its side: a +z ray runs along it, through most of its boxes."""
    x, y = np.meshgrid(np.arange(k), np.arange(k), indexing="ij")
    V = np.stack([rng.integers(0, 40, k * k), x.ravel(), y.ravel()], 1).astype(np.float32)
    a = (x[:-1, :-1] * k + y[:-1, :-1]).ravel()
    F = np.concatenate([np.stack([a, a + k, a + k + 1], 1), np.stack([a, a + k + 1, a + 1], 1)])
    return V, F.astype(np.int32)


@pytest.mark.parametrize("n", [32767, 32768, 32769])
def test_long_walks(n):
    import paper_2605_01536_gb300 as gwn
    rng = np.random.default_rng(n)
    V, F = rough_field(150, rng)
    Q = gen.queries_uniform_bbox(V, n, rng)
    Q[:64] = V[rng.integers(0, len(V), 64)] - np.float32([0, 0, 50])   # rays through vertices
    Q[64:128] = V[rng.integers(0, len(V), 64)]
    q = torch.from_numpy(Q).cuda()
    with gwn.Mesh(V, F) as m:
        _, chi = m.query(q)
        whole = m.counters()
    with gwn.Mesh(V, F) as m:
        parts = torch.cat([m.query(q[i:i + 5000])[1] for i in range(0, n, 5000)])
        split = m.counters()
    assert torch.equal(chi, parts)
    assert whole["error_flags"] == split["error_flags"] == 0
    assert whole["exact_edge"] == split["exact_edge"] > 0 and whole["exact_plane"] == split["exact_plane"] > 0
    sel = np.concatenate([np.arange(128), rng.choice(n, 100, replace=False)])
    assert np.array_equal(chi.cpu().numpy()[sel], oracle.reference(V, F, Q[sel])["chi"])
