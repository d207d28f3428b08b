"""The library's device-memory pool: results over streams and threads, and memory given back."""
import subprocess
import sys
import threading

import numpy as np
import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CHILD = """
import torch, gen
import paper_2605_01536_gb300 as gwn
mesh, rng = gen.displaced_soup(6, 3)
q = torch.from_numpy(gen.queries_uniform_bbox(mesh.V, 300_000, rng)).cuda()
with gwn.Mesh(mesh.V, mesh.F) as m:      # loads the kernels
    m.query(q)
torch.cuda.synchronize()
torch.cuda.empty_cache()
before = torch.cuda.mem_get_info()[0]
ms = [gwn.Mesh(mesh.V, mesh.F) for _ in range(3)]
for m in ms:
    m.query(q)
torch.cuda.synchronize()
held = before - torch.cuda.mem_get_info()[0]
for m in ms:
    m.close()
torch.cuda.empty_cache()
print(held, before - torch.cuda.mem_get_info()[0])
"""


def test_pool_is_given_back():
    out = subprocess.run([sys.executable, "-c", CHILD], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    held, kept = map(int, out.stdout.split())
    assert held > 0 and kept <= 4 << 20, (held, kept)


def test_threads_and_streams_share_the_pool():
    import paper_2605_01536_gb300 as gwn
    mesh, rng = gen.displaced_soup(5, 4)
    Q = [gen.queries_uniform_bbox(mesh.V, 20_000 + 777 * i, rng) for i in range(4)]
    with gwn.Mesh(mesh.V, mesh.F) as m:
        ref = [tuple(t.cpu() for t in m.query(torch.from_numpy(q).cuda())) for q in Q]
        bad = []

        def work(i):
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                q = torch.from_numpy(Q[i]).cuda()
                for _ in range(20):
                    w, chi = m.query(q)
                    with gwn.Mesh(mesh.V[:3], np.array([[0, 1, 2]], np.int32)) as small:
                        small.query(q[:10].contiguous())
                s.synchronize()
                if not (torch.equal(w.cpu(), ref[i][0]) and torch.equal(chi.cpu(), ref[i][1])):
                    bad.append(i)

        ts = [threading.Thread(target=work, args=(i,)) for i in range(4)]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
    assert not bad
