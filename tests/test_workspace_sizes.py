"""Workspace sizes of the calls whose products run on digits (16 bytes an
entry): the digits are formed a part at a time, so a workspace does not grow
with them beyond a few GB."""
import ctypes as C
import os

import pytest

GB = 1 << 30


@pytest.fixture(scope="module")
def L():
    from paper_1312_6838_gb300 import _lib, build
    if not os.path.exists(_lib.LIB_PATH):
        build.build()
    return _lib


def _size(L, op, dt, m, n, l, k):
    o = L.default_opts()
    return L.load().css_workspace_size(op, dt, m, n, l, k, 0, C.byref(o))


@pytest.mark.parametrize("m,n,l", [(4096, 65536, 256), (4096, 8000000, 1024), (8000000, 1000, 100), (10, 1 << 30, 1)])
def test_lowrank(L, m, n, l):
    assert 0 < _size(L, L.CSS_OP_LOWRANK, L.CSS_F64, m, n, l, l) <= 4 * GB
