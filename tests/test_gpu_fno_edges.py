"""GPU: the network at the ends of the range of the spectral branch inside a block: 32 retained
modes (the largest shared-memory request; on 64^2 all of them below the Nyquist index) and
2048 fields (the last count before the plans' transforms take over), against the FP64 oracle."""
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


@pytest.mark.parametrize("width,modes,n,batch", [
    (8, 32, 64, 2),
    (8, 31, 128, 1),
    (8, 32, 256, 1),
    (8, 33, 128, 1),   # one mode too many: the plans' transforms
    (32, 3, 32, 64),   # 2048 fields
    (32, 3, 32, 65),   # 2080: the plans' transforms
])
def test_forward_and_gradients_vs_oracle(width, modes, n, batch):
    # the tolerances of the gradient tests (single-precision sums against exact ones)
    cfg = FO.Config(width, 1, modes, 5)
    rng = np.random.default_rng(n + modes)
    p = FO.init_params(cfg, seed=modes).astype(np.float32)
    p += 0.05 * rng.standard_normal(p.size).astype(np.float32) / width
    a = rng.standard_normal((batch, 2, n, n)).astype(np.float32)
    t = rng.standard_normal((batch, n, n)).astype(np.float32)
    net = fch.FNO(width, 1, modes, 5)
    net.set_params(p)
    y = torch.empty((batch, n, n), dtype=torch.float32, device=DEV)
    at = torch.tensor(a, device=DEV)
    net.forward(at, y)
    loss = net.backward(torch.tensor(t, device=DEV))
    yr = FO.forward(p, a.astype(np.float64), cfg)
    G, R = cfg.unpack(net.grads()), cfg.unpack(FO.backward(p, a.astype(np.float64), t.astype(np.float64), cfg))
    assert np.linalg.norm(y.cpu().numpy() - yr) <= 2e-5 * np.linalg.norm(yr)
    assert abs(loss - np.mean((yr - t) ** 2)) <= 1e-4 * np.mean((yr - t) ** 2)
    for name in R:
        assert np.linalg.norm(G[name] - R[name]) <= 2e-4 * max(np.linalg.norm(R[name]), 1e-6), name
    net.close()
