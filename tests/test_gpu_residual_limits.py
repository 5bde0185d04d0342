"""The residual near FP32's limits: an entry of the gradient beyond the type's
range is an infinity of its sign, and a residual beyond FP32's range is still a
number of the FP64 loss.

The gradient of the columns outside S is 2 g R, rounded once.  Scaling A and g
by powers of two changes no digit of any product, so it is exactly 2^(e + q)
times the one at scale 1, or infinite."""
import pytest
import torch

import css_inputs as ci
from tests.gpu_helpers import dev_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("e,q", [(60, 66), (40, 90), (100, 28)])
def test_gradient_beyond_the_range_is_infinite(dtype, e, q):
    from paper_1312_6838_gb300 import css
    m, n, k = 130, 300, 12
    A, _ = dev_matrix(ci.lowrank_uv(m, n, k, 0.5, 821), dtype)

    def grad(X, g):
        X = X.detach().requires_grad_()
        css.residual(X, list(range(k))).backward(torch.tensor(g, device="cuda"))
        return X.grad
    got = grad(A * 2.0 ** e, 2.0 ** q)
    ref = (grad(A, 1.0).double() * 2.0 ** (e + q)).to(dtype)
    assert torch.isinf(ref[:, k:]).any() and torch.isfinite(ref[:, k:]).any()
    assert torch.equal(got[:, k:], ref[:, k:])
    assert not torch.isnan(got).any()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_residual_beyond_fp32(dtype, sign):
    """a = M (-1, 1, 1, 1) against (1, 1, 1, 1): r = M (-3/2, 1/2, 1/2, 1/2),
    whose first entry is beyond 2^128; ||r||^2 = 3 M^2."""
    from paper_1312_6838_gb300 import css
    M = 0.75 * 2.0 ** 128
    A = torch.zeros((3, 4), dtype=dtype, device="cuda").t()
    A[:, 0] = 1.0
    A[:, 1] = sign * M
    A[0, 1] = -sign * M
    loss = css.residual_error(A, [0])
    # (products and their difference from A in pairs of FP32 values)
    assert abs(loss - 3 * M * M) <= 2.0 ** -40 * M * M, loss
    X = A.detach().requires_grad_()
    css.residual(X, [0]).backward()
    g = X.grad[:, 1].double().cpu()
    assert g[0].item() == -sign * float("inf")
    assert torch.all((g[1:] - sign * M).abs() <= 2.0 ** -24 * M), g   # (2^-24: M is a number of either type)
    assert torch.all(X.grad[:, 2] == 0.0)
