"""CPU model of the index arithmetic of the passes built for a grid size
(csrc/fch_reg.cuh): natural slots at both ends of a transform, and the column pair with
column N - kx conjugated."""
import numpy as np
import pytest


def _fft_reg(x, ppt):
    """Forward transform on natural slots: thread t holds x[t + tps m], m < ppt; every
    stage reads and (the last one) writes slots of its own thread only."""
    n = len(x)
    tps, lp = n // ppt, 3 if ppt == 8 else 2
    v = np.array([[x[t + tps * m] for m in range(ppt)] for t in range(tps)])
    ns, rem = 1, int(np.log2(n))
    while rem:
        lr = min(lp, rem)
        R = 1 << lr
        nb = ppt // R
        k = np.arange(R)
        dft = np.exp(-2j * np.pi * np.outer(k, k) / R)
        buf = np.full(n, np.nan, dtype=complex)
        for t in range(tps):
            for b in range(nb):
                j = t + b * tps
                y = dft @ (v[t, b + nb * k] * np.exp(-2j * np.pi * k * (j % ns) / (ns * R)))
                v[t, b + nb * k] = y
                d = (j // ns) * ns * R + j % ns
                if ns * R == n:
                    assert np.array_equal(d + ns * k, t + tps * (b + nb * k))  # natural again
                buf[d + ns * k] = y
        if ns * R < n:
            assert not np.isnan(buf).any()
            v = np.array([[buf[t + tps * m] for m in range(ppt)] for t in range(tps)])
        ns, rem = ns * R, rem - lr
    return np.array([v[i % tps, i // tps] for i in range(n)])


@pytest.mark.parametrize("n", [64, 128, 256, 512, 1024, 2048])
@pytest.mark.parametrize("ppt", [4, 8])
def test_natural_slots_give_the_dft(n, ppt):
    rng = np.random.default_rng(n + ppt)
    x = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    X = _fft_reg(x, ppt)
    assert np.abs(X - np.fft.fft(x)).max() < 1e-12 * n
    # the inverse as conj, forward, conj
    assert np.abs(np.conj(_fft_reg(np.conj(X), ppt)) / n - x).max() < 1e-12


@pytest.mark.parametrize("n", [64, 128])
def test_column_pairs_with_a_conjugated_column(n):
    # two real fields a, b as z = a + i b; after the rows, column kx and the conjugate of
    # column N - kx transform along y to Z(kx, ky) and conj Z(N - kx, -ky): the split gives
    # the half spectra A, B at the same index, and the packed columns go back to z
    rng = np.random.default_rng(n)
    a, b = rng.standard_normal((2, n, n))
    A, B = np.fft.fft2(a), np.fft.fft2(b)  # [ky][kx]
    rows = np.fft.fft(a + 1j * b, axis=1)
    back = np.empty_like(rows)
    k = np.arange(n)
    for kx in range(1, n // 2):
        z0, w1 = _fft_reg(rows[:, kx], 4), _fft_reg(np.conj(rows[:, n - kx]), 4)
        Ah, Bh = 0.5 * (z0 + w1), (z0 - w1) / 2j
        assert np.allclose(Ah, A[:, kx]) and np.allclose(Bh, B[:, kx])
        o0 = np.conj(Ah + 1j * Bh)  # conj, forward, conj
        o1 = np.conj(Ah) + 1j * np.conj(Bh)  # column N - kx comes back without the last conj
        back[:, kx], back[:, n - kx] = np.conj(_fft_reg(o0, 4)) / n, _fft_reg(o1, 4) / n
    for c, kx in ((0, 0), (1, n // 2)):  # the columns that pair with themselves
        w = _fft_reg(np.conj(rows[:, kx]) if c else rows[:, kx], 4)
        zk, zm = w[k], w[-k % n]
        za, zb = (np.conj(zk), zm) if c else (zk, np.conj(zm))
        Ah, Bh = 0.5 * (za + zb), (za - zb) / 2j  # item k of column 0, -k of column N/2
        item = -k % n if c else k
        assert np.allclose(Ah, A[item, kx]) and np.allclose(Bh, B[item, kx])
        o = Ah + 1j * Bh
        back[:, kx] = _fft_reg(o, 4) / n if c else np.conj(_fft_reg(np.conj(o), 4)) / n
    assert np.allclose(back, rows)
    # the pair-layout slot of a natural index is a bijection
    slot = [2 * e if e < n // 2 else 1 if e == n // 2 else 2 * (n - e) + 1 for e in range(n)]
    assert sorted(slot) == list(range(n))


@pytest.mark.parametrize("logn", [6, 7, 8])
def test_two_point_stages_from_the_radix4_table(logn):
    # radix-2 stages on two points a thread, their factors taken from the table of radix-4
    # stages (one of radix 2 at its end where log2 n is odd), against numpy's transform
    from paper_2006_04784_gb300 import fch
    n = 1 << logn
    tw = fch.stage_twiddles(n, 2)
    tps = n // 2
    x = np.random.default_rng(n).standard_normal(2 * n).view(complex)
    v = np.stack([x[:tps], x[tps:]], axis=1)
    for s in range(logn):
        ns = 1 << s
        buf = np.full(n, np.nan, dtype=complex)
        for t in range(tps):
            b = v[t, 1]
            if s % 2 == 0 and s > 0:
                b *= tw[ns - 4 + (0 if s + 1 == logn else ns) + (t & (ns - 1))]
            elif s % 2:
                nh = ns >> 1
                if s > 1:
                    b *= tw[nh - 4 + (t & (nh - 1))]
                if t & nh:
                    b *= -1j
            d = ((t >> s) << (s + 1)) + (t & (ns - 1))
            buf[d], buf[d + ns] = v[t, 0] + b, v[t, 0] - b
        v = np.stack([buf[:tps], buf[tps:]], axis=1)
    out = np.concatenate([v[:, 0], v[:, 1]])
    assert np.abs(out - np.fft.fft(x)).max() < 1e-13 * n
