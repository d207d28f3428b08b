"""The hierarchy's truncation against the margin that makes labels exact.

The expansions a query takes may together be off by at most half the mesh's
classify_margin (the other half is FP32 rounding's).  A margin far below what the
expansions can hold must therefore leave the boundary to the direct sum: the same bits
as the mesh configured for it.
"""
import numpy as np
import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 100_003


def both(config, n=N):
    """w by the mesh's own rule and by the direct sum."""
    import paper_2605_01536_gb300 as gwn
    mesh, rng = gen.displaced_soup(6, 9)
    q = torch.from_numpy(gen.queries_uniform_bbox(mesh.V, n, rng)).cuda()
    with gwn.Mesh(mesh.V, mesh.F, config=config) as m, \
            gwn.Mesh(mesh.V, mesh.F, config={**config, "queries_per_thread": 4}) as d:
        return m.query(q)[0], d.query(q)[0]


def test_margin_below_the_expansions():
    w, wd = both({"classify_margin": 1e-9})
    assert torch.equal(w, wd)


@pytest.mark.parametrize("margin", [1e-5, 1e-4, 1e-2])
def test_margin_the_expansions_hold(margin):
    w, wd = both({"classify_margin": margin})
    assert not torch.equal(w, wd)   # the hierarchy was taken
    # half the margin, and FP32 rounding between the two (the library's 1e-6 each)
    assert torch.max(torch.abs(w - wd)).item() <= margin / 2 + 2e-6
