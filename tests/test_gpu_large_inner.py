"""Products from digits whose inner dimension is beyond a grid's 65535 blocks
of 64 (4,194,240) and beyond what one 64-bit sum holds (2^25 products of the
largest digits): the embedding and the residual of tall matrices, the Gram
matrix of long rows, FP64 selections of few rows."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def _randn(*shape, seed, dtype=torch.float64):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(*shape, generator=g, device="cuda", dtype=dtype)


@pytest.mark.parametrize("l,n", [(1, 4194241), (3, 4200001), (20, 5000000)])
def test_lowrank_of_long_rows(l, n):
    from paper_1312_6838_gb300 import css
    W = _randn(l, n, seed=n)
    r = css.lowrank(W, l)
    ref = torch.linalg.eigvalsh(W @ W.t()).flip(0)
    tol = 4 * (n + l) * U * float(W.square().sum())   # the Gram route's resolution
    assert float((r.sigma.square() - ref).abs().max()) <= tol
    err = (r.V.t() @ r.V - torch.eye(l, device="cuda", dtype=torch.float64)).abs().max()
    assert float(err) <= 1e-10
    rec = (r.Uw * r.sigma) @ r.V.t()
    assert float((rec - W).abs().max()) <= 1e-9


def test_gram_of_equal_digits():
    """2^26 products of the largest digit: 2^26 * 2^-6 is the exact sum."""
    from paper_1312_6838_gb300 import css
    W = torch.full((1, 1 << 26), 0.125, dtype=torch.float64, device="cuda")
    assert float(css.lowrank(W, 1, want_V=False).sigma[0]) == 2.0 ** 10


def test_lowrank_with_more_rows_of_q_than_columns():
    """U~ = Q U^(W) takes Q in parts; a workspace sized without Q's rows (m = 0)
    takes smaller ones, with the same result."""
    import ctypes as C

    from paper_1312_6838_gb300 import _lib as L, css
    l, n, m, k = 70, 300, 200001, 70
    W, Q = _randn(l, n, seed=1), _randn(l, m, seed=2).t()
    r = css.lowrank(W, k, Q)
    assert float((r.U - Q @ r.Uw).abs().max()) <= 4 * l * U * float(Q.abs().max()) * l ** 0.5
    lib, o = L.load(), L.default_opts()
    size = lib.css_workspace_size(L.CSS_OP_LOWRANK, L.CSS_F64, 0, n, l, k, 0, C.byref(o))
    ws = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
    U2 = torch.empty((k, m), dtype=torch.float64, device="cuda").t()
    sig = torch.empty(k, dtype=torch.float64, device="cuda")
    p = lambda t: C.c_void_p(t.data_ptr())
    code = lib.css_lowrank(p(W), n, p(Q), m, m, n, l, k, p(sig), p(U2), m, C.c_void_p(0), n, C.c_void_p(0),
                           C.c_void_p(0), C.c_void_p((ws.data_ptr() + 255) // 256 * 256), size, C.byref(o),
                           C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert code == 0 and torch.equal(U2, r.U)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("m,n,l", [(4194241, 5, 2), (4300001, 9, 4), (40000, 3000, 20), (700000, 300, 130)])
def test_embedding_and_residual_of_tall_columns(dtype, m, n, l):
    from paper_1312_6838_gb300 import css
    A = _randn(n, m, seed=m, dtype=dtype).t()
    S = list(range(1, 1 + l))
    X = A.double()
    Q, R = torch.linalg.qr(X[:, S])
    sg = torch.sign(torch.diagonal(R))
    Q, R = Q * sg, R * sg[:, None]
    emb = css.embed(A, S)
    W = Q.t() @ X
    # sums of m terms on both sides (the reference's round)
    assert float((emb.Q - Q).abs().max()) <= 1e-12
    assert float((emb.W - W).abs().max()) <= 1e-8
    E = X - Q @ W
    E[:, S] = 0.0
    Ag = A.detach().requires_grad_()
    loss = css.residual(Ag, S)
    loss.backward()
    u = 2.0 ** -53 if dtype == torch.float64 else 2.0 ** -24
    ref = float(E.square().sum())
    assert abs(float(loss.detach()) - ref) <= (1e-10 + 2 * u) * ref
    # (the last two sizes: columns, and columns and rows, in several parts)
    G = 2 * E
    G[:, S] = -2 * (E @ torch.linalg.solve_triangular(R, W, upper=True).t())
    assert float((Ag.grad.double() - G).abs().max()) <= (1e-10 + 8 * u) * float(G.abs().max())


def test_embedding_of_equal_digits():
    """A column of 2^26 ones: Q is 2^-13 throughout and W 2^13, exactly."""
    from paper_1312_6838_gb300 import css
    A = torch.ones(1, 1 << 26, dtype=torch.bfloat16, device="cuda").t()
    emb = css.embed(A, [0])
    assert float(emb.W[0, 0]) == 2.0 ** 13
    assert float(emb.Q.min()) == float(emb.Q.max()) == 2.0 ** -13


@pytest.mark.parametrize("m,n", [(5, 4194241), (3, 20000000), (9001, 300)])
def test_fp64_selection_of_few_long_rows(m, n):
    """(9001 rows: C's digits in two parts)"""
    from paper_1312_6838_gb300 import css
    A = _randn(n, m, seed=m).t()
    a, b = css.select(A, 2), css.select(A, 2, init_path=1)
    # (among millions of columns in a few dimensions the best are tied to the
    # last bits: the picks are compared through the error they leave)
    assert float((a.trace - b.trace).abs().max()) <= 8 * (m + n) * U * float(a.trace[0])
