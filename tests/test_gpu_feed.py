"""The greedy kernel's ways of feeding its products (greedy.cu): loads into
registers, the fused step's ring of asynchronous copies (FP32 with at least
256 KB of A per CTA) and the short rows of C (a CTA per problem, more problems
than CTAs).  They form the same sums in the same order, so one problem gives
the same bits through each of them: alone in one CTA, in a batch whose average
keeps to the register loads, and in a batch of its like."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

CTAS = 152
# fewer rows than a vector, one row step exactly and one more, row ends past
# the last whole vector, rows of C on both sides of the short-row limit
ROWS = [1, 2, 3, 4, 5, 7, 8, 9, 64, 127, 128, 129, 255, 256, 257, 511, 513, 960, 1023, 1919, 1920, 1921, 2047, 2050]


@pytest.fixture(scope="module")
def css():
    from paper_1312_6838_gb300 import css as c
    return c


def _problem(css, m, n, k, dtype, seed, rank_one=False):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((m, k)) @ rng.standard_normal((k, n)) + 0.01 * rng.standard_normal((m, n))
    if rank_one:
        X[:, 1:] = X[:, :1]   # the selection ends early
    return css.to_colmajor(torch.from_numpy(X).to(dtype).cuda()), min(k, m, n)


def _edges(css, dtype):
    """Problems of at least 256 KB in FP32 with ragged numbers of columns."""
    return [_problem(css, m, 65536 // m + 3 + 5 * i, 6, dtype, i, i % 5 == 4) for i, m in enumerate(ROWS)]


def _same(a, b):
    assert a.n_sel == b.n_sel
    assert torch.equal(a.indices, b.indices)
    assert torch.equal(a.trace[: a.n_sel + 1], b.trace[: b.n_sel + 1])


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float64])
def test_feeds_give_the_same_bits(css, dtype):
    edges = _edges(css, dtype)
    # a single FP64 problem has its own initial scores; init_path = 1 gives the batch's
    path = 1 if dtype == torch.float64 else 0
    alone = [css.select(A, k, grid_ctas=1, init_path=path) for A, k in edges]
    tiny = [_problem(css, 3 + i % 9, 2 + i % 13, 2, dtype, 1000 + i) for i in range(600)]
    # the tiny problems bring the average per CTA below the ring's line
    mixed = edges + tiny
    got = css.select_batched([A for A, _ in mixed], [k for _, k in mixed])
    for a, b in zip(alone, got):
        _same(a, b)
    alike = edges * (2 * CTAS // len(edges) + 1)
    got = css.select_batched([A for A, _ in alike], [k for _, k in alike])
    for i, b in enumerate(got):
        _same(alone[i % len(edges)], b)


@pytest.mark.parametrize("m,n,k", [(515, 60011, 9), (2048, 20000, 8), (3000, 15001, 5)])
def test_ring_over_many_ctas_is_repeatable(css, m, n, k):
    """More units than warps, drawn in any order: the same bits each time, and
    the trace against residual_error, which forms the residual anew (1e-4 of
    it: Theorem 1's recursion in FP32)."""
    A, k = _problem(css, m, n, k, torch.float32, m)
    a, b = css.select(A, k), css.select(A, k)
    _same(a, b)
    for t in (1, k):
        direct = css.residual_error(A, a.indices[:t])
        assert abs(a.trace[t].item() - direct) <= 1e-4 * direct + 1e-5 * a.trace[0].item()
