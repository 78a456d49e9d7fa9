"""CPU: which launches take the passes built for a grid size."""
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
