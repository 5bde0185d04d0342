"""B = A Omega with FP32 accumulation on 128-row tiles (project.cu) against FP64,
at the edges of its tiles, chunks and slices."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("m,n,r", [(1, 1, 1), (3, 15, 2), (127, 129, 31), (128, 16, 32), (129, 2049, 33),
                                   (255, 4097, 64), (131, 1000, 65), (257, 999, 128), (65, 5001, 129),
                                   (9, 8191, 257)])
def test_project_tiles(dtype, m, n, r):
    from paper_1312_6838_gb300 import css
    rng = np.random.default_rng(m * 7 + n + r)
    lda = m + 3   # columns that start on no 16-byte boundary
    buf = torch.from_numpy(rng.standard_normal((n, lda))).to(dtype).cuda()
    A = buf[:, :m].t()
    Om = torch.from_numpy(rng.standard_normal((r, n))).to(dtype).cuda().t()
    B = css.project(A, Om).double()
    exact = A.double() @ Om.double()
    size = A.double().abs() @ Om.double().abs()
    # a chain of n products and at most 32 partial sums in FP32: (n + 32) u
    assert torch.all((B - exact).abs() <= (n + 33) * 2.0 ** -24 * size)
