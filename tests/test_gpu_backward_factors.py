"""css.residual's gradient reuses the forward pass's Q, W and L^-1
(css_residual_backward_factors): the same bits as css_residual_backward, which
forms them itself."""
import ctypes as C

import pytest
import torch

import css_inputs as ci
from tests.gpu_helpers import dev_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.bfloat16])
@pytest.mark.parametrize("m,n,k,ld", [(65, 130, 7, 65), (129, 257, 33, 136), (300, 500, 140, 300)])
def test_gradient_is_the_same_bits(dtype, m, n, k, ld):
    from paper_1312_6838_gb300 import _lib as L, css
    A, _ = dev_matrix(ci.lowrank_uv(m, n, min(m, 2 * k), 0.05, 31 + k), dtype, ld=ld)
    S = torch.randperm(n, generator=torch.Generator().manual_seed(k))[:k].to(torch.int32).cuda()
    X = A.detach().requires_grad_()
    loss = css.residual(X, S)
    loss.backward(torch.tensor(2.5, dtype=loss.dtype, device="cuda"), retain_graph=True)
    first = X.grad.clone()
    X.grad = None
    loss.backward(torch.tensor(2.5, dtype=loss.dtype, device="cuda"))   # the factors are only read
    lib, o = L.load(), L.default_opts()
    dt = {torch.float64: L.CSS_F64, torch.float32: L.CSS_F32, torch.bfloat16: L.CSS_BF16}[dtype]
    nbytes = lib.css_workspace_size(L.CSS_OP_BACKWARD, dt, m, n, 0, k, 0, C.byref(o))
    buf = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    ws = C.c_void_p((buf.data_ptr() + 255) // 256 * 256)
    dA = css.empty_colmajor(m, n, dtype)
    l = torch.empty(1, dtype=torch.float64, device="cuda")
    code = lib.css_residual_backward(C.c_void_p(A.data_ptr()), dt, m, n, A.stride(1), C.c_void_p(S.data_ptr()), k, 2.5,
                                     C.c_void_p(dA.data_ptr()), m, C.c_void_p(l.data_ptr()), ws, nbytes, C.byref(o),
                                     C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert code == 0
    assert torch.equal(first, dA) and torch.equal(X.grad, dA)
    with torch.no_grad():
        assert torch.equal(css.residual(A, S), loss)
    assert torch.equal(loss.double(), l[0].to(loss.dtype).double())
