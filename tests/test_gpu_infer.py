"""Network outputs on both sides of the switch to several tiles per block, and with a last
tile of one query: the same bits as in short calls, within 0.05 of the FP64 network."""
import numpy as np
import pytest

import gen
from oracle import mlp as ref

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extra", [0, 1, 127, 128, 129, 128 * 152 * 3 + 1])
def test_predict(extra):
    import paper_2605_01536_gb300 as gwn
    n = 3 * 128 * torch.cuda.get_device_properties(0).multi_processor_count + extra
    rng = np.random.default_rng(extra)
    P = {}
    for name, shape in ref._SHAPES:
        scale = np.sqrt(2.0 / shape[1]) if name.startswith("W") else (0.2 if name == "w5" else 0.05)
        P[name] = rng.normal(scale=scale, size=shape)
    p = ref.pack(P).astype(np.float32)
    box = np.array([-1, -1, -1, 1, 1, 1], np.float32)
    q = rng.uniform(-1, 1, (n, 3)).astype(np.float32)
    mesh = gen.small_cap(3, 0.8)
    with gwn.Mesh(mesh.V, mesh.F) as m:
        m.set_surrogate_params(p, box)
        d = torch.from_numpy(q).cuda()
        w = m.surrogate_predict(d)
        parts = torch.cat([m.surrogate_predict(d[i:i + 20001]) for i in range(0, n, 20001)])
    assert torch.equal(w, parts)
    # BF16 features and activations over five layers of He-scaled weights: outputs of order 1,
    # about ten roundings of 2^-9 each in the mean square, six deviations
    y, _ = ref.forward(p.astype(np.float64), box, q[-300:])
    assert np.max(np.abs(w.cpu().numpy()[-300:] - y)) <= 0.05
