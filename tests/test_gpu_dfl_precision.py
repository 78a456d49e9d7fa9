"""GPU: the double-float functions of the pointwise and ETD stages against extended
precision, at the accuracy of the format."""
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

LD = np.longdouble


def _split(x):
    """x rounded to double-float, as extended precision"""
    h = x.astype(np.float32)
    return h.astype(LD) + (x - h.astype(LD)).astype(np.float32).astype(LD)


def _args(lo, hi, n=50000):
    return _split(np.random.default_rng(11).uniform(lo, hi, n).astype(LD)).astype(np.float64)


def _rms(x):
    return float(np.sqrt((x * x).mean()))


@pytest.mark.parametrize("lo,hi", [(-0.01, 0.01), (-0.1, 0.1), (0.1, 1.0), (-1.0, -0.1), (-5.0, 0.0), (-20.0, 0.0), (0.0, 80.0)])
def test_exp_and_expm1_round_once(lo, hi):
    # the error is that of rounding the exact value to double-float: what remains (2^-52 and
    # below, expm1 near 0.1 2^-51) adds at most a twentieth to its rms and a bit to its largest
    x = _args(lo, hi)
    xt = torch.tensor(x, device="cuda:0")
    out = [torch.empty_like(xt) for _ in range(2)]
    torch.cuda.synchronize()
    f = fch.lib().fch_debug_dfl_exp
    f.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p, C.c_long, C.c_void_p]
    assert f(xt.data_ptr(), out[0].data_ptr(), out[1].data_ptr(), x.size, None) == 0
    for o, ref in zip(out, (np.exp(x.astype(LD)), np.expm1(x.astype(LD)))):
        err, own = o.cpu().numpy().astype(LD) / ref - 1, _split(ref) / ref - 1
        assert _rms(err) <= 1.05 * _rms(own)
        assert np.abs(err).max() <= 2.0 ** -48


def _point(phi, q, x):
    xt = torch.tensor(x, device="cuda:0")
    out = torch.empty((3, x.size), dtype=torch.float64, device="cuda:0")
    torch.cuda.synchronize()
    f = fch.lib().fch_debug_dfl_point
    f.argtypes = [C.c_void_p, C.c_int, C.c_void_p, C.c_void_p, C.c_long, C.c_void_p]
    p = fch.params_default(q)
    assert f(C.byref(p), phi, xt.data_ptr(), out.data_ptr(), x.size, None) == 0
    return out.cpu().numpy().astype(LD)


@pytest.mark.parametrize("lo,hi,t1,t2", [(1e-4, 0.2, -50.5, -50.5), (0.199, 0.201, -49.0, -46.0), (0.2, 1.0, -49.0, -46.8),
                                         (1.0, 30.0, -49.0, -47.8), (30.0, 1e4, -49.3, -48.0)])
def test_etd_phi(lo, hi, t1, t2):
    # rms bounds (bits): the series to its 2^-51; the quotients to half a bit above what they
    # measure, e^z - 1 - z having lost 1 / (z/2) of its size below z = 2
    z = -np.exp(_args(np.log(lo), np.log(hi)))
    z = _split(z.astype(LD)).astype(np.float64)
    ez, p1, p2 = _point(1, 0.0, z)
    z = z.astype(LD)
    if hi <= 1.0:
        r1, r2 = np.zeros_like(z), np.zeros_like(z)
        fact = np.cumprod(np.arange(1, 24).astype(LD))
        for j in range(20, -1, -1):
            r1, r2 = r1 * z + 1 / fact[j], r2 * z + 1 / fact[j + 1]
    else:
        r1, r2 = np.expm1(z) / z, (np.expm1(z) - z) / (z * z)
    ok = np.exp(z) > 1e-25  # (below, the low word leaves the range of a float)
    assert np.abs(ez / np.exp(z) - 1)[ok].max() <= 2.0 ** -48 if ok.any() else True
    assert _rms(p1 / r1 - 1) <= 2.0 ** t1
    assert _rms(p2 / r2 - 1) <= 2.0 ** t2


@pytest.mark.parametrize("q,bits", [(0.2, (-45.9, -46.8, -46.9)), (0.5, (-45.9, -46.8, -46.3))])
def test_regularised_well(q, bits):
    # W, W', W'' over the range of a solution: rms bounds (bits of the rms value) a third of a
    # bit above what renormalised sums and the quotient (u - b_-) / eps measure
    p = fch.params_default(q)
    u = _args(-1.6, 1.6)
    got = _point(0, q, u)
    c = lambda v: _split(np.array([v], dtype=LD))[0]  # noqa: E731  (constants as the library holds them)
    u = u.astype(LD)
    v, w = u - c(p.b_minus), u - c(p.b_plus)
    x = v / c(p.eps)
    e = np.exp(-np.abs(x))
    s, th = 2 * e / (1 + e * e), np.sign(x) * (1 - e * e) / (1 + e * e)
    A, A1 = v * v / 2 + c(p.q * p.eps) * (1 - s), v + c(p.q) * s * th
    A2 = 1 + c(p.q / p.eps) * s * (2 * s * s - 1)
    g3, c3 = c(p.gamma / 3.0), c(0.5 * (3.0 * p.b_plus - p.b_minus))
    Bq, B1 = w * w / 2 + g3 * (u - c3), w + g3
    for a, r, t in zip(got, (A * Bq, A1 * Bq + A * B1, A2 * Bq + 2 * A1 * B1 + A), bits):
        assert _rms(a - r) <= 2.0 ** t * _rms(r), t
