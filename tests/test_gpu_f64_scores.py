"""FP64 initial scores from integer digits (init_f64.cu) against the FP64 tiles
(init_path = 1), and the workspace without the digits."""
import ctypes as C

import numpy as np
import pytest
import torch

import css_inputs as ci

pytestmark = pytest.mark.gpu


def _problem(m, n, pad, seed):
    X = ci.lowrank_uv(m, n, max(1, min(m, n) // 2), 0.05, seed)
    X *= 10.0 ** np.random.default_rng(seed).uniform(-4, 4, n)   # columns of very different size
    buf = torch.zeros((n, m + pad), dtype=torch.float64, device="cuda")
    buf[:, :m] = torch.from_numpy(X.T.copy()).cuda()
    return buf[:, :m].t()


@pytest.mark.parametrize("m,n,pad", [(1, 3, 0), (2, 129, 1), (63, 64, 0), (65, 127, 2), (127, 300, 1), (128, 128, 0),
                                     (129, 2049, 3), (257, 16385, 0)])
def test_scores_match_the_fp64_tiles(m, n, pad):
    from paper_1312_6838_gb300 import css
    A = _problem(m, n, pad, m + n)
    a = css.select(A, 1, diag=True)
    b = css.select(A, 1, diag=True, init_path=1)
    assert torch.equal(a.sel, b.sel)
    # f after one pick: sums of at most m + n products each, of which none
    # exceeds ||A||^2 ||a_i||^2
    scale = a.trace[0] * A.square().sum(0)
    assert torch.all((a.diag_f - b.diag_f).abs() <= 16 * (m + n) * 2.0 ** -53 * scale + 1e-300)
    assert abs(a.trace[1] - b.trace[1]) <= 16 * (m + n) * 2.0 ** -53 * a.trace[0]


def test_equal_columns_tie():
    from paper_1312_6838_gb300 import css
    A = _problem(200, 900, 0, 5)
    A[:, 700] = A[:, 31]
    A[:, 31:700] *= 0.5
    A[:, 31] = A[:, 700]
    r = css.select(A, 1, diag=True, forced=[0])
    assert r.diag_f[31] == r.diag_f[700]


def test_least_workspace():
    """A workspace without room for the digits is still taken: the FP64 tiles."""
    from paper_1312_6838_gb300 import _lib as L, css
    m, n, k = 100, 700, 5
    A = _problem(m, n, 0, 9)
    lib, o = L.load(), L.default_opts()
    full = lib.css_workspace_size(L.CSS_OP_SELECT, L.CSS_F64, m, n, 0, k, 0, C.byref(o))
    small = full - 40 * 1024 * 1024   # the digits' partial sums alone take 39.8 MB
    ws = torch.empty(full + 256, dtype=torch.uint8, device="cuda")
    base = (ws.data_ptr() + 255) // 256 * 256
    got = []
    for size in (small, full):
        sel = torch.empty(k, dtype=torch.int32, device="cuda")
        trace = torch.empty(k + 1, dtype=torch.float64, device="cuda")
        ns = torch.zeros(1, dtype=torch.int32, device="cuda")
        p = lambda t: C.c_void_p(t.data_ptr())
        code = lib.css_select(p(A), L.CSS_F64, m, n, m, k, p(sel), p(trace), p(ns), C.c_void_p(0), C.c_void_p(base),
                              size, C.byref(o), C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert code == 0, L.status_string(code)
        got.append((sel, trace))
    tiles, digits = css.select(A, k, init_path=1), css.select(A, k)
    assert torch.equal(got[0][1], tiles.trace) and torch.equal(got[0][0], tiles.sel)
    assert torch.equal(got[1][1], digits.trace) and torch.equal(got[1][0], digits.sel)
