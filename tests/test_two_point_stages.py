"""CPU model of the transforms of two points a thread (csrc/fch_reg.cuh, reg_stage2): radix-8
stages level by level over the natural slots, with the library's twiddle table."""
import numpy as np
import pytest

from paper_2006_04784_gb300 import fch


@pytest.mark.parametrize("logn", [6, 7, 8])
def test_levels_of_radix8_stages_give_the_dft(logn):
    n = 1 << logn
    tw = fch.stage_twiddles(n, 3)
    x = np.random.default_rng(n).standard_normal(2 * n).view(complex)
    t = np.arange(n // 2)
    v = [x[: n // 2].copy(), x[n // 2:].copy()]

    def trade(w0, w1):
        buf = np.full(n, np.nan, dtype=complex)
        buf[w0], buf[w1] = v
        assert not np.isnan(buf).any()  # every slot written once
        v[0], v[1] = buf[t], buf[t + n // 2]

    def sums():
        v[0], v[1] = v[0] + v[1], v[0] - v[1]

    s, rem = 0, logn
    while rem:
        lr = min(3, rem)
        nb, ns = n >> lr, 8 ** s
        j, c, last = t & (nb - 1), t >> (logn - lr), (ns << lr) == n
        if ns > 1:
            base = ns - 8 + (j & (ns - 1))
            v[0] = np.where(c > 0, v[0] * tw[np.where(c > 0, base + (c - 1) * ns, 0)], v[0])
            v[1] = v[1] * tw[base + (c + (1 << lr >> 1) - 1) * ns]
        sums()
        if lr >= 2:
            q = 2 * (c & 1) + 4 * (c >> 1) if lr == 3 else 2 * c
            trade(j + q * nb, j + (q + 1) * nb)
            v[1] = np.where(c & 1, -1j * v[1], v[1])
            sums()
        if lr == 3:
            q = (c & 1) + 4 * (c >> 1)
            trade(j + q * nb, j + (q + 2) * nb)
            v[1] = v[1] * np.exp(-0.25j * np.pi * c)
            sums()
        if not last:
            d = ((j >> (3 * s)) << (3 * s + lr)) + (j & (ns - 1)) + c * ns
            trade(d, d + 4 * ns)
        s, rem = s + 1, rem - lr
    assert np.abs(np.concatenate(v) - np.fft.fft(x)).max() < 1e-13 * n
