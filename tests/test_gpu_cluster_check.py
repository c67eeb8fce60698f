"""The check that the cluster kernels make before they read or write a peer's shared
memory: a launch whose clusters are not of the expected size records CFET_ECUDA."""

import ctypes as C

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size,expected", [(4, 4), (8, 8), (2, 2), (1, 4), (2, 4), (8, 4), (1, 16)])
def test_cluster_check(size, expected):
    pytest.importorskip("torch")
    from paper_1102_5071_gb300 import _capi
    from paper_1102_5071_gb300.build import build
    build()
    st = C.c_int32(-1)
    assert _capi.load().cfet_selftest_cluster_check(size, expected, C.byref(st)) == _capi.CFET_OK
    assert st.value == (0 if size == expected else _capi.CFET_ECUDA)
