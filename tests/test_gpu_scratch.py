"""Scratch of large calls over the boundary hierarchy: bounded, whatever the split of the walks."""
import numpy as np
import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["gradient", "query"])
def test_scratch_of_split_walks(call):
    """300,000 queries: 21 MB of order and results, and at most 128 MiB of partial sums (a split into
    as many parts at once: 300 MB for the gradient).  Memory the library holds after the call is
    what it took (its pool keeps up to 1 GiB)."""
    import paper_2605_01536_gb300 as gwn
    mesh, rng = gen.displaced_soup(6, 9)
    q = torch.from_numpy(gen.queries_uniform_bbox(mesh.V, 300_000, rng)).cuda()
    with gwn.Mesh(mesh.V, mesh.F) as m:
        getattr(m, call)(q[:20_000].contiguous())
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        held = torch.cuda.memory_reserved()
        getattr(m, call)(q)
        torch.cuda.synchronize()
        grown = before - torch.cuda.mem_get_info()[0] - (torch.cuda.memory_reserved() - held)
    assert grown <= 176 << 20, grown


@pytest.mark.parametrize("call", ["gradient", "query"])
def test_slices_give_the_same_bits(call):
    """Enough queries for several slices of the partial sums against each query in a smaller call of
    the same split (a query's sums do not depend on the slice it falls into)."""
    import paper_2605_01536_gb300 as gwn
    mesh, rng = gen.displaced_soup(6, 9)
    n = 300_000
    Q = gen.queries_uniform_bbox(mesh.V, n, rng)
    q = torch.from_numpy(Q).cuda()
    run = lambda m, x: m.gradient(x) if call == "gradient" else m.query(x)[0]
    with gwn.Mesh(mesh.V, mesh.F) as m:
        g = run(m, q)
        perm = torch.randperm(n, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
        assert torch.equal(run(m, q[perm].contiguous()), g[perm])
