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


@pytest.mark.parametrize("dt", ["CSS_F64", "CSS_F32", "CSS_BF16"])
@pytest.mark.parametrize("m,n,k", [(4096, 65536, 256), (16384, 262144, 128), (16384, 524288, 128), (512, 8000000, 16),
                                   (8000000, 512, 16), (1 << 26, 2, 1)])
def test_gradient(L, dt, m, n, k):
    # A_S, Q and R W^T of m x k doubles and W, beside at most 6 GB
    size = _size(L, L.CSS_OP_BACKWARD, getattr(L, dt), m, n, 0, k)
    assert 0 < size <= 8 * (4 * m * k + k * n) + 6 * GB


@pytest.mark.parametrize("m,n,l", [(4096, 65536, 256), (8000000, 512, 16), (1000000, 2000, 1000), (1 << 26, 2, 1)])
def test_embedding(L, m, n, l):
    assert 0 < _size(L, L.CSS_OP_EMBED, L.CSS_BF16, m, n, 0, l) <= 8 * 4 * m * l + 6 * GB


@pytest.mark.parametrize("m,n,l", [(4096, 65536, 256), (4096, 8000000, 1024), (8000000, 1000, 100), (10, 1 << 30, 1)])
def test_lowrank(L, m, n, l):
    assert 0 < _size(L, L.CSS_OP_LOWRANK, L.CSS_F64, m, n, l, l) <= 4 * GB


@pytest.mark.parametrize("m,n", [(8, 4190000), (8, 16000000), (100, 10000000), (1000, 1000000), (100000, 10000)])
def test_fp64_selection(L, m, n):
    # C, its digits and C A of a part, the score state, and the digits of a part of A
    size = _size(L, L.CSS_OP_SELECT, L.CSS_F64, m, n, 0, 4)
    assert 0 < size <= 8 * m * m + 100 * n + min(32 * (m + 128) ** 2, 17 * GB) + 2 * GB
