"""css_residual_backward's small calls form their products in FP64 instead of
digits: both sides of the rule, at the edges of the kernel's 8 x 8 tiles and
chunks of 32, against the oracle with the adjoint's own tolerances."""
import pytest
import torch

import css_inputs as ci
from oracle import css_oracle as O
from tests import test_gpu_loss_range as loss_range
from tests.gpu_helpers import dev_matrix, gradient_entry_errors, gradient_tolerances

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.bfloat16])
@pytest.mark.parametrize("m,n,k,ld", [
    (9, 17, 1, 9), (33, 65, 7, 40), (31, 300, 9, 31), (64, 129, 32, 64), (300, 40, 33, 301), (40, 4096, 3, 40),
    (2049, 40, 5, 2049), (128, 256, 16, 128), (129, 257, 16, 136),
    # digits: a longer sum, more multiply-adds
    (40, 4097, 3, 40), (257, 1300, 31, 257),
])
def test_against_the_oracle(dtype, m, n, k, ld):
    from paper_1312_6838_gb300 import css
    A, vals = dev_matrix(ci.lowrank_uv(m, n, k, 1e-2, 700 + m), dtype, ld=ld)
    S = O.greedy_css(vals, k, tau_rel=1e-10).S
    L_ref, G_ref = O.residual_gradient(vals, S)
    X = A.detach().requires_grad_()
    loss = css.residual(X, S)
    loss.backward()
    assert abs(loss.item() - L_ref) <= 1e-6 * L_ref
    assert abs(css.residual_error(A, S) - L_ref) <= 1e-9 * L_ref
    G = X.grad.double().cpu().numpy()
    tol, tol_S = gradient_tolerances(vals, S, G_ref, dtype)
    rest, sel = gradient_entry_errors(G, G_ref, S, tol, tol_S)
    assert rest <= 1.0 and sel <= 1.0, (rest, sel)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float64])
@pytest.mark.parametrize("e", [80, 60, -73, -100])
def test_loss_of_digits_at_any_scale(dtype, e, monkeypatch):
    monkeypatch.setattr(loss_range, "SHAPE", (260, 3100, 13))
    loss_range.test_loss_at_any_scale(dtype, e)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("e,q", [(60, 66), (100, 28)])
def test_gradient_of_digits_beyond_the_range(dtype, e, q):
    """See test_gpu_residual_limits.py."""
    from paper_1312_6838_gb300 import css
    m, n, k = 130, 6500, 12
    A, _ = dev_matrix(ci.lowrank_uv(m, n, k, 0.5, 823), dtype)

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
def test_residual_of_digits_beyond_fp32(dtype, sign):
    from paper_1312_6838_gb300 import css
    M = 0.75 * 2.0 ** 128
    A = torch.zeros((5000, 4), dtype=dtype, device="cuda").t()
    A[:, 0] = 1.0
    A[:, 1] = sign * M
    A[0, 1] = -sign * M
    loss = css.residual_error(A, [0])
    assert abs(loss - 3 * M * M) <= 2.0 ** -40 * M * M, loss
    X = A.detach().requires_grad_()
    css.residual(X, [0]).backward()
    g = X.grad[:, 1].double().cpu()
    assert g[0].item() == -sign * float("inf")
    assert torch.all((g[1:] - sign * M).abs() <= 2.0 ** -24 * M), g
    assert torch.all(X.grad[:, 2:] == 0.0)
