"""GPU: the passes built for a size with two or four points a thread round no more than the
generic kernels of eight: F(u) of both against extended precision."""
import numpy as np
import pytest

from paper_2006_04784_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2006_04784_gb300 import build as B  # noqa: E402

B.build()
from paper_2006_04784_gb300 import fch  # noqa: E402

LD = np.longdouble
DEV = torch.device("cuda:0")


def _rhs(u, p):
    """F(u) = Lap mu(u) at q = 0 in the precision of u (L = 4 pi)"""
    LD, n = u.dtype.type, len(u)
    e2, k = LD(p.eps) ** 2, LD(0.5) * np.concatenate([np.arange(n // 2), np.arange(-n // 2, 0)]).astype(LD)
    k2 = k[:, None] ** 2 + k[None, :] ** 2
    F, R = np.fft.fft2, lambda z: np.fft.ifft2(z).real
    v, w = u - LD(p.b_minus), u - LD(p.b_plus)
    g3, c3 = LD(p.gamma) / 3, (3 * LD(p.b_plus) - LD(p.b_minus)) / 2
    A, Bq, B1 = v * v / 2, w * w / 2 + g3 * (u - c3), w + g3
    W1, W2 = v * Bq + A * B1, Bq + 2 * v * B1 + A
    lu = R(-k2 * F(u))
    om = e2 * lu - W1
    mu = -e2 * k2 * F(om) + F(-W2 * om + e2 * LD(p.eta1) * lu - LD(p.eta2) * W1)
    return R(-k2 * mu)


def _errors(n, prec, seeds, dtype):
    err = {0: [], -1: []}
    for seed in range(seeds):
        u = I.circle_bilayer(n, noise=0) + 1e-2 * np.random.default_rng(seed).uniform(-1, 1, (n, n))
        if prec == 1:
            u = u.astype(np.float32).astype(np.float64)
        ut, ref = torch.tensor(u, device=DEV), None
        for tile in (0, -1):
            p = fch.params_default(0.0, prec=prec, tile_row=tile, tile_col=tile)
            if ref is None:
                ref = _rhs(u.astype(dtype), p)
            with fch.Context(n, p) as c:
                out = torch.empty_like(ut)
                torch.cuda.synchronize()
                c.rhs_device(ut, out)
                c.synchronize()
            d = out.cpu().numpy().astype(dtype) - ref
            err[tile].append(float(np.sqrt((d * d).sum() / (ref * ref).sum())))
    return np.mean(err[0]), np.mean(err[-1])


@pytest.mark.parametrize("n,prec", [(64, 0), (128, 0), (64, 1), (128, 1), (256, 1), (64, 2), (128, 2), (256, 2)])
def test_two_points_a_thread(n, prec):
    # the mean error over six fields is known to about 1 % (its seeds differ by 2-3 %)
    built, generic = _errors(n, prec, 6, LD)
    assert built <= 1.04 * generic


@pytest.mark.parametrize("n", [512, 1024])
def test_four_points_a_thread_in_double_float(n):
    # two fields: the mean error over a million points is known to half a per cent
    built, generic = _errors(n, 2, 2, np.float64)
    assert built <= 1.01 * generic
