"""Record exchange of the persistent kernels: sums over all CTAs' records are exact
and every word of a record carries the exchange's tag or, where a short record leaves
the second pair of words as it was, one not so old that the stored 16 bits of it could
repeat, with the kernels' record widths mixed, with one slot left to short records for
thousands of exchanges, and across the repetition."""

import ctypes as C

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [2, 31, 33, 152, 160, 161, 200])  # 160 records are held in registers
@pytest.mark.parametrize("first,n", [(1, 40), (65510, 60), (3 * 65536 + 65533, 20), (4 * 65536, 9), (1, 68000)])
def test_exchange_words_and_sums(grid, first, n):
    pytest.importorskip("torch")
    from paper_1102_5071_gb300 import _capi
    from paper_1102_5071_gb300.build import build
    build()
    wrong = (C.c_int64 * 2)(-1, -1)
    assert _capi.load().cfet_selftest_exchange(grid, first, n, wrong) == _capi.CFET_OK
    assert list(wrong) == [0, 0]
