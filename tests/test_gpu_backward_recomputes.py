"""css.residual's gradient forms the k x k factor and what follows from it anew
from A and S: the forward pass leaves nothing behind but the two."""
import pytest
import torch

import css_inputs as ci
from tests.gpu_helpers import dev_matrix

pytestmark = pytest.mark.gpu

M, N, K = 300, 500, 140


def _problem():
    A, _ = dev_matrix(ci.lowrank_uv(M, N, 2 * K, 0.05, 17), torch.float64)
    return A, torch.randperm(N, generator=torch.Generator().manual_seed(3))[:K].to(torch.int32).cuda()


def test_forward_keeps_no_products():
    from paper_1312_6838_gb300 import css
    A, S = _problem()
    X = A.detach().requires_grad_()
    css.residual(X, S).backward()
    X.grad = None
    before = torch.cuda.memory_allocated()
    loss = css.residual(X, S)
    # Q, W and L^-1 would be 1 MB
    assert torch.cuda.memory_allocated() - before <= 64 * 1024
    loss.backward()


def test_gradient_is_that_of_the_matrix_it_finds():
    from paper_1312_6838_gb300 import css
    A, S = _problem()
    B = A * 2.0 + 1.0
    X = A.detach().clone(memory_format=torch.preserve_format).requires_grad_()
    loss = css.residual(X, S)
    X.data.copy_(B)
    loss.backward()
    Y = B.detach().requires_grad_()
    css.residual(Y, S).backward()
    assert torch.equal(X.grad, Y.grad)
