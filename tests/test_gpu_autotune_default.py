"""GPU: the tuner times the default column kernel that plans run."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2006_04784_gb300 import build as B  # noqa: E402

B.build()
from paper_2006_04784_gb300 import fch  # noqa: E402


def test_single_precision_1024_columns_are_the_plans():
    # a plan's transform of 16 fields is one launch each of the rows and columns over eight
    # pairs, as the tuner times them; with another column kernel the sum is a third above it
    stream = torch.cuda.Stream()
    x = torch.randn((16, 1024, 1024), device="cuda:0")
    X = torch.empty((16, 513, 1024), dtype=torch.complex64, device="cuda:0")
    torch.cuda.synchronize()
    fch.autotune_reset()
    plan = fch.FFTPlan(1024, 1, stream=stream)
    us = []
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        for _ in range(20):
            plan.r2c(x, X)
        b.record(stream)
        b.synchronize()
        us.append(a.elapsed_time(b) * 50.0)
    plan.status()
    plan.close()
    t = fch.autotune(1024, 1)
    fch.autotune_reset()
    assert t["row_default_us"] + t["col_default_us"] <= 1.15 * min(us)
