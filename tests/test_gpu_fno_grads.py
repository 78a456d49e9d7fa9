"""GPU: every gradient of the network against the FP64 oracle at channel counts off the
weight-gradient kernel's 32 x 32 tiles, odd batches, and an input array off the 16-byte
alignment of its wide loads."""
import numpy as np
import pytest

from oracle import fno_oracle as FO

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2006_04784_gb300 import build as B  # noqa: E402

B.build()
from paper_2006_04784_gb300 import fch  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("width,layers,modes,proj,n,batch,shift", [
    (8, 1, 3, 5, 16, 1, 0),      # outputs below a tile, one short run of points
    (8, 2, 3, 33, 32, 3, 1),     # one column over a tile, the input one float off alignment
    (16, 2, 8, 63, 64, 5, 3),
    (32, 1, 16, 64, 32, 3, 0),   # whole tiles
    (8, 1, 4, 128, 128, 2, 2),   # four tiles of rows
    (32, 2, 16, 64, 256, 1, 0),
])
def test_gradients_vs_oracle_off_the_tiles(width, layers, modes, proj, n, batch, shift):
    # the tolerances of the gradient tests (single-precision sums against exact ones)
    cfg = FO.Config(width, layers, modes, proj)
    p = FO.init_params(cfg, seed=n + proj).astype(np.float32)
    p += 0.05 * np.random.default_rng(3).standard_normal(p.size).astype(np.float32) / width
    rng = np.random.default_rng(n + batch)
    a = rng.standard_normal((batch, 2, n, n)).astype(np.float32)
    t = rng.standard_normal((batch, n, n)).astype(np.float32)
    net = fch.FNO(width, layers, modes, proj)
    net.set_params(p)
    store = torch.empty(a.size + 4, dtype=torch.float32, device=DEV)
    at = store[shift:shift + a.size].view(a.shape)
    at.copy_(torch.tensor(a))
    y = torch.empty((batch, n, n), dtype=torch.float32, device=DEV)
    net.forward(at, y)
    loss = net.backward(torch.tensor(t, device=DEV))
    g = net.grads()
    ref = FO.backward(p, a.astype(np.float64), t.astype(np.float64), cfg)
    yr = FO.forward(p, a.astype(np.float64), cfg)
    assert np.linalg.norm(y.cpu().numpy() - yr) <= 2e-5 * np.linalg.norm(yr)
    assert abs(loss - np.mean((yr - t) ** 2)) <= 1e-4 * np.mean((yr - t) ** 2)
    G, R = cfg.unpack(g), cfg.unpack(ref)
    for name in R:
        assert np.linalg.norm(G[name] - R[name]) <= 2e-4 * max(np.linalg.norm(R[name]), 1e-6), name
    net.close()
