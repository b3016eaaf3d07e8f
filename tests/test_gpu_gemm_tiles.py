"""Parity of the GEMM where its persistent CTAs take several tiles each: odd
numbers of two-k-block steps (the steps of consecutive tiles are numbered
through), every tile width, code rows a tensor map cannot take (q = 3 with k an
odd multiple of 64) and scale rows that allow no vector load."""
import pytest

import oracle  # noqa: F401  (the reference that run_case compares with)
from paper_2607_08779_gb300 import inputs, sss

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


@pytest.mark.parametrize("n,k,m,chain", [
    (1024, 1152, 256, 5 * 8),     # 9 steps of 8 MMAs over the four accumulators of a 64-token tile, or two
    (4096, 14336, 512, 56 * 8),   # 112 steps: K split in two, or the two of a 128-token tile
    (512, 4096, 40, 8 * 8),
])
def test_gemm_chains_of_accumulation_are_divided(n, k, m, chain):
    # the weights of the symmetric q = 2 grid are exact in fp16, so what is left is
    # the truncation of the sums: up to 2^-24 of the partial sum per MMA, half of it
    # on average.  The partial sum grows as the square root of its terms, so a
    # chain of c MMAs is off by 2/3 c 2^-25 of its result
    qt = sss.sss_quantize(inputs.student_t_weights_cuda(n, k, 3, outliers=False), 2, 32,
                          sss.GRID_SIGNED_SYM)
    x = inputs.normal_bf16_cuda((m, k), 4)
    ref = x.double() @ sss.sss_dequantize(qt).double().T
    err = ((sss.sss_gemm(qt, x).double() - ref).norm() / ref.norm()).item()
    assert err <= 2 / 3 * chain * 2.0**-25
