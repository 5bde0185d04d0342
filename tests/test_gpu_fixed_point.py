"""Products from digits hold a row's entries relative to its largest one, so
operands whose inner index runs over very different sizes are balanced first:
a power of two per inner index, taken from the diagonal of the Gram matrix,
moves from one operand to the other.  Matrices whose rows (or columns) differ
by many orders of magnitude, against FP64 arithmetic."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.mark.parametrize("m,n,big", [(100, 300, 1.0), (100, 300, 1e8), (65, 257, 1e15), (300, 2100, 1e15)])
def test_fp64_scores_beside_an_outlying_row(m, n, big):
    """One row holds entries of size `big` in every seventh column and zeros
    elsewhere.  The other columns' scores do not see them.  After one forced
    pick among them, f against the FP64 tiles: sums of at most m + n products
    of row norms s_r, |f_i| errors below (m + n) u (sum_r s_r |a_ri|)^2 each
    (two initial scores and their updates: factor 8)."""
    from paper_1312_6838_gb300 import css
    rng = np.random.default_rng(n)
    X = rng.standard_normal((m, n))
    X[3] = 0.0
    X[3, ::7] = big
    A = css.to_colmajor(torch.from_numpy(X).cuda())
    a = css.select(A, 1, diag=True, forced=[1]).diag_f.cpu().numpy()
    b = css.select(A, 1, diag=True, forced=[1], init_path=1).diag_f.cpu().numpy()
    s = np.linalg.norm(X, axis=1)
    tol = 8 * (m + n) * U * (s @ np.abs(X)) ** 2
    worst = np.max(np.abs(a - b) / tol)
    print(f"f beside {big:g}: {worst:.3g} of the tolerance")
    assert worst <= 1.0, worst


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("l", [128, 129, 200])
def test_basis_of_graded_columns(dtype, l):
    """A_S with columns over eight decades: Q = orth(A_S) does not depend on
    their sizes.  Against Householder QR of the columns at one scale; both
    within 8 l u cond^2 (the normal equations square the condition of the
    scaled columns, which is all that counts), entrywise."""
    from paper_1312_6838_gb300 import css
    rng = np.random.default_rng(l)
    X = rng.standard_normal((400, l)) * np.exp2(np.rint(-26.0 * rng.permutation(l) / (l - 1)))
    A = css.to_colmajor(torch.from_numpy(X).to(dtype).cuda())
    X = A.double().cpu().numpy()
    X = X / np.exp2(np.rint(np.log2(np.abs(X).max(0))))
    Q, R = np.linalg.qr(X)
    Q *= np.sign(np.diag(R))
    got = css.embed(A, list(range(l))).Q.cpu().numpy()
    tol = 8 * l * U * np.linalg.cond(X) ** 2
    worst = np.abs(got - Q).max()
    print(f"Q of graded columns, l = {l}: {worst:.3g}, tolerance {tol:.3g}")
    assert worst <= tol
