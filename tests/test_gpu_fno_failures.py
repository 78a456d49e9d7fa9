"""GPU: what a forward pass that fails on the host (work arrays beyond the device's memory)
leaves behind."""
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

DEV = torch.device("cuda:0")
ENOMEM, ESTATE = 2, 7


def _net():
    net = fch.FNO(16, 1, 16, 16)
    rng = np.random.default_rng(4)
    net.set_params((0.1 * rng.standard_normal(net.num_params)).astype(np.float32))
    a = torch.tensor(rng.standard_normal((1, 2, 128, 128)).astype(np.float32), device=DEV)
    return net, a, torch.empty((1, 128, 128), device=DEV)


def _fail(net, a, y):
    # 2048^2 x 4096 samples: the first array alone takes two terabytes, so the call ends
    # before it reads or launches anything
    st = fch.lib().fch_fno_forward(net._h, 4096, 2048, C.c_void_p(a.data_ptr()), C.c_void_p(y.data_ptr()))
    assert st == ENOMEM


@pytest.mark.parametrize("first", ["fp32", "tensor cores", "none"])
def test_backward_is_refused_after_a_failed_forward(first):
    net, a, y = _net()
    if first == "fp32":
        net.forward(a, y)
        net.backward(y)
    elif first == "tensor cores":
        net.set_bf16(2)
        net.forward(a, y)
        net.set_bf16(0)
    _fail(net, a, y)
    loss = C.c_double(-1.0)
    assert fch.lib().fch_fno_backward(net._h, C.c_void_p(y.data_ptr()), C.byref(loss)) == ESTATE
    assert loss.value == -1.0
    torch.cuda.synchronize()
    net.close()


def test_a_failed_forward_leaves_no_error_for_the_next_call():
    # neither the library's next launch check nor another library's finds the allocation's error
    net, a, y = _net()
    net.forward(a, y)
    ref = y.clone()
    _fail(net, a, y)
    net.set_bf16(1)  # launches a kernel and checks
    net.set_bf16(0)
    _fail(net, a, y)
    net.set_params(net.params())
    net.forward(a, y)
    assert torch.equal(y, ref)
    net.backward(ref)
    _fail(net, a, y)
    assert float((torch.ones(8, device=DEV) + 1).sum()) == 16.0
    net.close()
