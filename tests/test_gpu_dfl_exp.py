"""GPU: the double-float exp and expm1 (the q > 0 well, the ETD phi functions) against
numpy's double ones over the ranges and edges of their branches."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2006_04784_gb300 import build as B  # noqa: E402

B.build()
from paper_2006_04784_gb300 import fch  # noqa: E402


def _eval(x):
    xt = torch.tensor(x, device="cuda:0")
    out = [torch.empty_like(xt) for _ in range(2)]
    torch.cuda.synchronize()
    f = fch.lib().fch_debug_dfl_exp
    f.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p, C.c_long, C.c_void_p]
    assert f(xt.data_ptr(), out[0].data_ptr(), out[1].data_ptr(), x.size, None) == 0
    return [o.cpu().numpy() for o in out]


@pytest.mark.parametrize("lo,hi", [(-1e-9, 1e-9), (-0.0109, 0.0109), (-0.36, 0.36), (-2.0, 2.0), (-20.0, 0.0), (-60.0, 20.0)])
def test_relative_error(lo, hi):
    # 2^-47 of the evaluation and 2^-49 |x| of the argument's own rounding to double-float
    x = np.random.default_rng(7).uniform(lo, hi, 20000)
    x = x.astype(np.float32).astype(np.float64) + (x - x.astype(np.float32)).astype(np.float32)
    ex, em = _eval(x)
    tol = 2.0 ** -46.5 * (1 + np.abs(x))
    assert (np.abs(ex / np.exp(x) - 1) <= tol).all()
    assert (np.abs(em / np.expm1(x) - 1) <= tol).all()


def test_edges():
    # underflow to zero (to -1), overflow, the argument zero, NaN; the branch points
    x = np.array([0.0, -0.0, -1e3, -1e9, -np.inf, 1e3, np.inf, np.nan, 0.35, -0.35, 88.0, -103.0])
    ex, em = _eval(x)
    assert ex[0] == 1 and ex[1] == 1 and em[0] == 0 and em[1] == 0
    assert (ex[2:5] == 0).all() and (em[2:5] == -1).all()
    assert not np.isfinite(ex[5:8]).any() and not np.isfinite(em[5:8]).any()
    assert np.allclose(ex[8:11], np.exp(x[8:11]), rtol=1e-13) and np.allclose(em[8:11], np.expm1(x[8:11]), rtol=1e-13)
    assert 0 <= ex[11] < 1e-44 and em[11] == -1
