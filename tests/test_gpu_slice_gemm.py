"""Products from integer digits on the tensor cores (csrc/slice_gemm.cu),
reached through css.embed (W = Q^T A): every entry against numpy's FP64
product of the device's own Q with A, at the edges of the kernel's tiles
(128 x 128 results, 16 and 64 inner indices, split-K) and over wide ranges.

Tolerance per entry: the FP64 reference's own bound (m + 2) 2^-53 sum|q||a|,
plus the kernel's, its final conversion (3 roundings) and its dropped digits
(36 terms below 2^-64 of the scaled row maxima, which are at most 4 times the
largest entries).
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def css():
    from paper_1312_6838_gb300 import css as c
    return c


def _check(css, A, S):
    emb = css.embed(A, S)
    Q, W = emb.Q.cpu().numpy(), emb.W.cpu().numpy()
    X = A.double().cpu().numpy()
    m = X.shape[0]
    ref = Q.T @ X
    own = 36 * m * 2.0 ** -64 * 16 * np.abs(Q).max(0)[:, None] * np.abs(X).max(0)[None, :]
    tol = (m + 2) * U * (np.abs(Q).T @ np.abs(X)) + 3 * U * np.abs(ref) + own
    assert (np.abs(W - ref) <= tol).all()


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.bfloat16])
@pytest.mark.parametrize("m,n,l,lda", [
    (1, 1, 1, 1), (15, 128, 1, 16), (16, 129, 7, 16), (17, 127, 16, 17), (63, 40, 33, 63), (64, 257, 64, 72),
    (65, 300, 65, 65), (129, 131, 127, 131), (200, 385, 128, 200), (333, 200, 129, 333), (1025, 150, 20, 1025),
    (4097, 260, 3, 4104), (520, 19500, 130, 520),
])
def test_product_at_tile_edges(css, dtype, m, n, l, lda):
    rng = np.random.default_rng(m * 7 + n)
    X = torch.from_numpy(rng.standard_normal((m, n))).to(dtype).cuda()
    _check(css, css.to_colmajor(X, ld=lda), list(rng.permutation(n)[:l]))


@pytest.mark.parametrize("dtype,spread", [(torch.float64, 30.0), (torch.float32, 6.0), (torch.bfloat16, 6.0)])
def test_product_over_a_wide_range(css, dtype, spread):
    """Entries over many binades, zero columns and a tiny one."""
    rng = np.random.default_rng(3)
    X = rng.standard_normal((300, 400)) * np.exp(spread * rng.standard_normal((300, 400)))
    X[:, 7] = 0.0
    X[:, 11] *= 2.0 ** -60
    _check(css, css.to_colmajor(torch.from_numpy(X).to(dtype).cuda()), [1, 5, 30, 200])


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_largest_digits_sum_exactly(css, dtype):
    """Every digit of A as large as it can be and of one sign: the
    accumulators run to the largest integers between two drains."""
    m = 5000
    X = np.full((m, 130), 127.0 / 255.0)
    X[:, 1::2] *= -1.0
    _check(css, css.to_colmajor(torch.from_numpy(X).to(dtype).cuda()), [0])


def test_non_finite_columns_as_fp64_arithmetic_gives_them(css):
    rng = np.random.default_rng(5)
    X = rng.standard_normal((70, 50))
    X[3, 20], X[4, 30], X[5, 31] = np.inf, np.nan, -np.inf
    A = css.to_colmajor(torch.from_numpy(X).cuda())
    emb = css.embed(A, [0, 1])
    Q, W = emb.Q.cpu().numpy(), emb.W.cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref = Q.T @ X
    assert np.array_equal(np.isnan(W), np.isnan(ref))
    inf = np.isinf(ref)
    assert inf.any() and np.array_equal(W[inf], ref[inf])
    ok = np.isfinite(ref)
    assert np.isfinite(W[ok]).all()
