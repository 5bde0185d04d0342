"""Products from digits whose inner dimension is beyond a grid's 65535 blocks
of 64 (4,194,240): the embedding and the residual of tall matrices, the Gram
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


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("m,n,l", [(4194241, 5, 2), (4300001, 9, 4)])
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
    G = 2 * E
    G[:, S] = -2 * (E @ torch.linalg.solve_triangular(R, W, upper=True).t())
    assert float((Ag.grad.double() - G).abs().max()) <= (1e-10 + 8 * u) * float(G.abs().max())


@pytest.mark.parametrize("m,n", [(5, 4194241), (3, 20000000)])
def test_fp64_selection_of_few_long_rows(m, n):
    from paper_1312_6838_gb300 import css
    A = _randn(n, m, seed=m).t()
    a, b = css.select(A, 2), css.select(A, 2, init_path=1)
    # (among millions of columns in a few dimensions the best are tied to the
    # last bits: the picks are compared through the error they leave)
    assert float((a.trace - b.trace).abs().max()) <= 8 * (m + n) * U * float(a.trace[0])
