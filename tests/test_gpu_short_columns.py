"""Columns so short that the fused step's split tiles have empty row chunks: a
team's CTAs take their first units turned by one from warp to warp (greedy.cu,
first_unit).  Whatever the team's size, every unit is taken once: the picks and
every column's final score state are those of a single CTA.

Tolerance: the recursions' rounding differs only through the team's partial
sums of the pivot, a few m eps of the column's norm a pick: 1e-10 and 1e-4
hold for FP64 and FP32 pivots with room; a unit missed or taken twice leaves
eight columns off by their share of the picks' directions, of order one."""
import pytest
import torch

import css_inputs as ci
from tests.gpu_helpers import dev_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,rows", [(torch.float64, (63, 64, 65, 192, 193)), (torch.float32, (127, 128, 384, 385)),
                                        (torch.bfloat16, (255, 768, 769))])
@pytest.mark.parametrize("tile", [2, 4, 8])
def test_every_unit_once(dtype, rows, tile):
    from paper_1312_6838_gb300 import css
    k = 6
    for m in rows:
        n = 131
        A, vals = dev_matrix(ci.lowrank_uv(m, n, 40, 0.3, 900 + m), dtype)
        one = css.select(A, k, grid_ctas=1, tile_cols=tile, diag=True)
        g0 = torch.from_numpy((vals ** 2).sum(0)).cuda()
        tol = 1e-10 if dtype == torch.float64 else 1e-4
        for ctas in (2, 3, 4, 7, 8, 16, 32):
            r = css.select(A, k, grid_ctas=ctas, tile_cols=tile, diag=True, forced=one.indices)
            assert r.indices.tolist() == one.indices.tolist()
            assert ((r.diag_g - one.diag_g).abs() <= tol * g0).all(), (m, ctas)
