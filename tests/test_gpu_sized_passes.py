"""GPU: the passes built for a grid size (tile 0) against the generic kernels (tile -1) at
every size and precision, on fields with every mode populated, and their transforms
against torch's at every size."""
import math

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

DEV = torch.device("cuda:0")
SIZES = [64, 128, 256, 512, 1024, 2048]


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("prec", [0, 1, 2])
def test_sized_passes_match_the_generic_kernels(n, prec):
    # both sides round a transform's sums differently: a few units of the pass precision
    # (2^-53, 2^-24, 2^-48) times log2 n a transform, some ten transforms, damped by the
    # solves; white noise fills every mode, the two self-paired columns among them
    tol = {0: 1e-12, 1: 3e-5, 2: 1e-11}[prec]
    u0 = I.circle_bilayer(n, noise=2e-2)
    for scheme in ("imex", "sav", "etd", "psd"):
        if prec == 1 and scheme == "psd":
            continue  # its tolerance lies below single precision
        out = []
        for tile in (0, -1):
            p = fch.params_default(0.2 if scheme == "etd" else 0.0, prec=prec, zero_stab_cap=1, tile_row=tile, tile_col=tile)
            with fch.Context(n, p) as ctx:
                ctx.set_state(u0)
                for dt in (1e-6, 2e-6, 1e-6):
                    ctx.step(scheme, dt)
                fixed = [ctx.get_state(), np.array([ctx.energy(), ctx.mass()])]
                # trials that keep the real-space fields (the direct row passes)
                if prec != 1:
                    ctx.set_state(u0)
                    st = ctx.run_adaptive(scheme, 1e-4, 1.0, max_attempts=6, raise_on_timeout=False)
                    fixed += [ctx.get_state(), np.array([st["t"], st["k_last"]])]
                out.append(fixed)
        for a, b in zip(*out):
            assert rel(a, b) < tol, (scheme, rel(a, b))


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("batch", [1, 5])
def test_sized_transforms_match_torch(n, prec, batch):
    # the tolerance of the transform parity tests (rounding of log2 n stages); an odd batch
    # ends with a field without a partner
    x = torch.randn((batch, n, n), dtype=torch.float32 if prec else torch.float64, device=DEV)
    X = torch.empty((batch, n // 2 + 1, n), dtype=torch.complex64 if prec else torch.complex128, device=DEV)
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    plan = fch.FFTPlan(n, prec)
    plan.r2c(x, X)
    plan.c2r(X, y)
    plan.status()
    ref = torch.fft.rfft2(x.double()).transpose(1, 2)
    tol = 2e-6 if prec else 1e-13
    assert (X - ref).abs().max() <= tol * ref.abs().max() * math.log2(n)
    assert (y - x).abs().max() <= tol * x.abs().max() * math.log2(n)
    plan.close()


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("scheme", ["imex", "sav"])
def test_mean_mode_is_kept_to_the_last_bit(prec, scheme):
    # u = u^n + (c/a)(u^n - u^{n-1}) at k = 0: a state without history keeps its mean exactly
    with fch.Context(64, fch.params_default(0.0, prec=prec, zero_stab_cap=1)) as ctx:
        ctx.set_state(I.circle_bilayer(64))
        m0 = ctx.mass()
        for dt in (1e-4, 3e-4, 1e-4, 7e-5):
            ctx.step(scheme, dt)
        assert ctx.mass() == m0


@pytest.mark.parametrize("n", [16, 128, 1024])
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("scheme", ["imex", "sav", "etd"])
def test_fused_fixed_steps_equal_single_steps(n, prec, scheme):
    # from the second step of a run on, the solve packs the next step's u*: the same bits as
    # steps of their own, whatever the length of the run and what went before it
    u0 = I.circle_bilayer(n, noise=1e-2)
    p = fch.params_default(0.0, prec=prec)
    with fch.Context(n, p) as a, fch.Context(n, p) as b:
        a.set_state(u0)
        b.set_state(u0)
        for m, dt in ((1, 2e-6), (2, 1e-6), (3, 1e-6), (4, 3e-6), (6, 3e-6)):
            for _ in range(m):
                a.step(scheme, dt)
            b.run_fixed(scheme, dt, m)
            assert np.array_equal(a.get_state(), b.get_state()), (m, dt)
