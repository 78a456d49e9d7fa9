"""CPU: which launches take the passes built for a grid size."""
import ctypes as C

import pytest

from paper_2006_04784_gb300 import fch


@pytest.mark.parametrize("xf", [0, 1])
@pytest.mark.parametrize("prec", [0, 1, 2])
def test_the_twiddle_table_a_pass_reads_decides(prec, xf):
    # every size from 64 up has built passes; without the radix-4 table (the transform that
    # allocates nothing keeps none) all but those of four points a thread remain
    f = fch.lib().fch_debug_built_pass
    for n in (16, 32, 64, 128, 256, 512, 1024, 2048):
        p = f(n, prec, xf, 1)
        assert p in ((2, 4, 8) if n >= 64 else (0,)), n
        assert f(n, prec, xf, 0) == (0 if p == 4 else p), n
    assert f(512, 0, xf, 0) == 8 and f(256, 0, xf, 0) == 0


@pytest.mark.parametrize("xf", [0, 1])
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("n", [64, 128, 256, 512, 1024, 2048])
def test_launches_cover_the_grid(n, prec, xf):
    out = (C.c_int * 8)()
    assert fch.lib().fch_debug_built_config(n, prec, xf, out) == 0
    ppt, rpb, row_threads, row_smem, ncol, col_blocks, col_threads, col_smem = out
    assert ppt == fch.lib().fch_debug_built_pass(n, prec, xf, 1)
    csz, tps = 8 if prec == 1 else 16, n // ppt
    assert n % rpb == 0 and row_threads == rpb * tps and row_threads % 32 == 0
    assert col_blocks * ncol == n and col_threads == ncol * tps and col_threads % 32 == 0
    assert max(row_threads, col_threads) <= 1024 and col_blocks <= 4096
    # a skewed sequence for every row and column of a block
    assert rpb * (n + n // 8) * csz <= row_smem <= 226 * 1024
    assert ncol * (n + n // 8) * csz <= col_smem <= 226 * 1024


@pytest.mark.parametrize("n", [16, 64, 256, 2048])
def test_index_maps(n):
    out = (C.c_int * (2 * n))()
    assert fch.lib().fch_debug_maps(n, out) == 0
    skew, slot = list(out[:n]), list(out[n:])
    assert sorted(set(skew)) == skew and skew[-1] < n + n // 8  # increasing, within a skewed sequence
    # pair p of the layout holds columns p and n - p (pair 0: 0 and n / 2)
    assert sorted(slot) == list(range(n))
    assert slot[0] == 0 and slot[n // 2] == 1
    assert all(slot[k] == 2 * k and slot[n - k] == 2 * k + 1 for k in range(1, n // 2))
