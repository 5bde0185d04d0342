"""The gradient of the selected columns where they are far larger than the
rest, as a greedy choice on graded data leaves them.  R is zero in those
columns, so they add nothing to R W^T, but they hold the largest entries of
W's rows: whatever precision is relative to a row's largest entry must not be
that of the result.

Tolerance per entry of dA_S = -2 (R W^T) L^-1 (entrywise absolute values of
the exact factors): the rounding of R to FP32, 2^-24 |R| |W|^T; R's own error,
(2^-46 + 4 k 2^-53 cond(A_S)^2) ||a_c|| in column c (products and their
difference from A in pairs of FP32 values, Q through the normal equations),
times |W|^T; both times |L^-1|; and the rounding of dA to its own type.
"""
import numpy as np
import pytest
import torch

from oracle import css_oracle as O
from tests.gpu_helpers import dev_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float64])
@pytest.mark.parametrize("m,n,k,c", [(96, 1024, 8, 1e2), (96, 1024, 8, 1e4), (130, 700, 30, 1e4), (200, 1500, 140, 1e3)])
def test_selected_columns_larger_than_the_rest(dtype, m, n, k, c):
    from paper_1312_6838_gb300 import css
    rng = np.random.default_rng(m + n)
    A_np = rng.standard_normal((m, n))
    S = [int(i) for i in rng.permutation(n)[:k]]
    A_np[:, S] *= c
    A, X = dev_matrix(A_np, dtype)
    _, G_ref = O.residual_gradient(X, S)
    Ag = A.detach().requires_grad_()
    css.residual(Ag, S).backward()
    G = Ag.grad.double().cpu().numpy()[:, S]
    u = {torch.float64: 2.0 ** -53, torch.float32: 2.0 ** -24, torch.bfloat16: 2.0 ** -8}[dtype]
    u_R = 2.0 ** -53 if dtype == torch.float64 else 2.0 ** -24
    Q, L = np.linalg.qr(X[:, S])   # L^T
    W = Q.T @ X
    R = X - Q @ W
    R[:, S] = 0.0
    kappa = np.linalg.cond(X[:, S])
    dR = np.broadcast_to((2.0 ** -46 + 4 * k * 2.0 ** -53 * kappa ** 2) * np.linalg.norm(X, axis=0), X.shape)
    tol = 2 * (u_R * np.abs(R) + dR) @ np.abs(W).T @ np.abs(np.linalg.inv(L).T) + u * np.abs(G_ref[:, S])
    worst = np.max(np.abs(G - G_ref[:, S]) / tol)
    print(f"dA_S {dtype} {m} x {n}, k = {k}, selected columns {c:g} times the rest: {worst:.3f} of the tolerance")
    assert worst <= 1.0, worst
