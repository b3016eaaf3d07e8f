"""Parity of the GEMM where its persistent CTAs take several tiles each: odd
numbers of two-k-block steps (the steps of consecutive tiles are numbered
through), every tile width, code rows a tensor map cannot take (q = 3 with k an
odd multiple of 64) and scale rows that allow no vector load."""
import pytest

import oracle  # noqa: F401  (the reference that run_case compares with)
from paper_2607_08779_gb300 import sss

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_gemm import run_case  # noqa: E402


@pytest.mark.parametrize("m", [1, 33, 65, 130, 270])
@pytest.mark.parametrize("q,g,k,grid", [
    (4, 32, 320, sss.GRID_SIGNED_SYM),    # 5 k-blocks: 3 steps, the last of one k-block
    (3, 64, 192, sss.GRID_ASYM),          # no code map, 3 scales per row
    (3, 32, 384, sss.GRID_UNSIGNED_SYM),  # 3 steps, 96-byte code tiles
    (2, 128, 384, sss.GRID_ASYM),         # 3 steps, one scale each
    (2, 64, 64, sss.GRID_SIGNED_SYM),     # a single k-block
    (4, 64, 128, sss.GRID_SIGNED_SYM),    # a single step
    (2, 32, 1152, sss.GRID_UNSIGNED_SYM),  # 9 steps
])
def test_gemm_several_tiles_per_cta(q, g, k, grid, m):
    # 157 row tiles: more than the SMs, the last one ragged
    run_case(20004, k, m, q, g, grid, 31 * q + g + k + m, tokens=[0, m // 2, m - 1])
