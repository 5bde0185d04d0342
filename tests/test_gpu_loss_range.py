"""The residual's loss is an FP64 number whatever the scale of A: entries whose
squares leave FP32's range are summed as any others.

Scaling A by a power of two changes no digit of any product, so the loss at
scale 2^e is 2^(2 e) times the loss at scale 1, but for the low parts of
entries below 2^-126 (2^-149 absolute, against residuals above 2^-108 here:
2^-41 relative, twice that in a square) and the sums' rounding (2^-46 each)."""
import ctypes as C

import pytest
import torch

import css_inputs as ci
from oracle import css_oracle as O
from tests.gpu_helpers import dev_matrix

pytestmark = pytest.mark.gpu

SHAPE = (200, 900, 12)


def _matrix(dtype):
    m, n, k = SHAPE
    A, vals = dev_matrix(ci.lowrank_uv(m, n, k, 0.05, 811), dtype)
    return A, vals, list(range(k))


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float64])
@pytest.mark.parametrize("e", [80, 60, -73, -100])
def test_loss_at_any_scale(dtype, e):
    from paper_1312_6838_gb300 import css
    A, vals, S = _matrix(dtype)
    one = css.residual_error(A, S)
    assert abs(one - O.reconstruction_error(vals, S)) <= 1e-7 * one
    got = css.residual_error(A * 2.0 ** e, S)   # (keeps the column-major strides)
    assert abs(got * 2.0 ** (-2 * e) - one) <= 2.0 ** -38 * one, (got, one)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_loss_of_columns_at_both_ends_of_the_range(dtype):
    """Half of the columns at 2^70, the others at 2^-90: the loss is that of
    the large ones; the large ones selected and exactly reproduced, it is that
    of the small ones."""
    from paper_1312_6838_gb300 import css
    m, n, k = 64, 40, 4
    A, vals = dev_matrix(ci.lowrank_uv(m, n, 20, 0.05, 812), dtype)
    A = A.clone(memory_format=torch.preserve_format)
    A[:, ::2] *= 2.0 ** 70
    A[:, 1::2] *= 2.0 ** -90
    X = A.double().cpu().numpy()
    S = [0, 2, 4, 6]
    ref = O.reconstruction_error(X, S)
    assert abs(css.residual_error(A, S) - ref) <= 1e-7 * ref
    # columns of one entry each: their residual is exactly zero
    A[:, ::2] = 0.0
    for j, c in enumerate(S):
        A[j, c] = 2.0 ** 70
        A[j, 1::2] = 0.0
    X = A.double().cpu().numpy()
    ref = float((X[:, 1::2] ** 2).sum())
    assert abs(css.residual_error(A, S) - ref) <= 1e-7 * ref


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_loss_beyond_fp32_is_infinite_there(dtype):
    """css.residual rounds to FP32: a loss above its range is +inf, not NaN."""
    from paper_1312_6838_gb300 import css
    A, _, S = _matrix(dtype)
    assert css.residual(A * 2.0 ** 80, S).item() == float("inf")
