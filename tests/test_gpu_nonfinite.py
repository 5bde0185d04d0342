"""Infinities and NaN in products from digits (csrc/slice_gemm.cu): reported or
passed on as FP64 arithmetic gives them, and never by a wait that runs out
while one thread restores them."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

BUDGET_NS = 20_000_000


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("m,n", [(300, 16384), (2304, 16384)])
def test_fp64_selection_reports_non_finite_data(m, n, bad):
    """C = A A^T of 2304 rows has more result tiles than the GPU has SMs, so a
    CTA that restores a row of its first tile has a second one waiting."""
    from paper_1312_6838_gb300 import _lib as L, css
    g = torch.Generator(device="cuda").manual_seed(m)
    A = torch.randn(n, m, generator=g, device="cuda", dtype=torch.float64).t()
    A[0, n // 2] = bad
    with pytest.raises(L.CssError) as ei:
        css.select(A, 2, spin_budget_ns=BUDGET_NS)
    assert ei.value.code == L.CSS_ERR_NONFINITE


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.bfloat16])
@pytest.mark.parametrize("m,n,l", [(520, 19600, 130), (700, 300, 17)])
def test_columns_of_the_embedding(dtype, m, n, l):
    """W = Q^T A with whole tiles of non-finite columns, unsplit and split
    products: every entry as FP64 arithmetic gives it where that is infinite
    or NaN, finite where that is finite."""
    from paper_1312_6838_gb300 import css
    rng = np.random.default_rng(m)
    X = rng.standard_normal((m, n))
    X[rng.integers(0, m, 90), 140 + np.arange(90)] = np.where(rng.random(90) < 0.5, np.inf, -np.inf)
    X[5, 150], X[6, 150] = np.inf, -np.inf
    X[rng.integers(0, m, 9), 260 + np.arange(9)] = np.nan
    A = css.to_colmajor(torch.from_numpy(X).to(dtype).cuda())
    emb = css.embed(A, list(range(l)))
    Q, W = emb.Q.cpu().numpy(), emb.W.cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref = Q.T @ A.double().cpu().numpy()
    fin = np.isfinite(ref)
    assert np.array_equal(np.isnan(W), np.isnan(ref))
    assert np.array_equal(W[np.isinf(ref)], ref[np.isinf(ref)])
    assert np.isfinite(W[fin]).all() and np.allclose(W[fin], ref[fin], rtol=0, atol=1e-11)


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_lowrank_reports_non_finite_data(bad):
    from paper_1312_6838_gb300 import _lib as L, css
    W = torch.randn(200, 30000, dtype=torch.float64, device="cuda")
    W[150, 29999] = bad
    with pytest.raises(L.CssError) as ei:
        css.lowrank(W, 5)
    assert ei.value.code == L.CSS_ERR_NONFINITE
