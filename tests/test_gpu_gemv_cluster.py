"""The batched GEMV for q = 2 and 4 (gemv_cluster.cu) at the sizes where its
split can go wrong: fewer steps than a cluster has CTAs, a k that the CTAs do
not divide, scale rows aligned to 16, 8 and 4 bytes, ragged rows, and enough
rows that the partial sums take several passes.  Integer dots and scales meet
in fp32, so the error is that of fp32 sums."""
import pytest

from paper_2607_08779_gb300 import inputs, sss

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_gemv import run_case  # noqa: E402

# fp32 sums of k <= 8192 products in any order: at most k 2^-24 relative to the
# sum of magnitudes, in practice sqrt(k) of it, against the largest output
TOL = 2e-5


@pytest.mark.parametrize("batch", [2, 8, 9, 16])
@pytest.mark.parametrize("q", [2, 4])
@pytest.mark.parametrize("n,k,g,grid", [
    (24, 256, 32, sss.GRID_SIGNED_SYM),   # less than a tile, 2 steps
    (33, 256, 128, sss.GRID_ASYM),        # scale rows of 4 bytes
    (100, 1280, 128, sss.GRID_SIGNED_SYM),  # 20-byte scale rows, 10 steps
    (65, 4352, 64, sss.GRID_ASYM),        # 136-byte scale rows, 34 steps
    (2000, 3328, 32, sss.GRID_UNSIGNED_SYM),  # 26 steps
])
def test_gemv_cluster_edges(n, k, g, grid, q, batch):
    run_case(n, k, q, g, grid, batch, n + k + g + q + batch, outliers=False, tol=TOL)


@pytest.mark.parametrize("q,grid,batch", [(4, sss.GRID_SIGNED_SYM, 16), (2, sss.GRID_ASYM, 5)])
def test_gemv_cluster_many_rows(q, grid, batch):
    n, k = 300_017, 256
    qt = sss.sss_quantize(inputs.student_t_weights_cuda(n, k, 7, outliers=False), q, 32, grid)
    x = inputs.normal_bf16_cuda((batch, k), 8)
    y = sss.sss_gemv(qt, x)
    ref = x.double() @ sss.sss_dequantize(qt).double().T
    assert ((y - ref).abs().amax(1) / ref.abs().amax(1)).max().item() <= TOL


def test_gemv_cluster_large_activations():
    # 30000 fits the fp16 operand whatever the field's position
    n, k = 64, 512
    w = inputs.student_t_weights_cuda(n, k, 9, outliers=False)
    for q in (2, 4):
        qt = sss.sss_quantize(w, q, 32, sss.GRID_SIGNED_SYM)
        x = inputs.normal_bf16_cuda((3, k), 10)
        x[1] *= 8000.0
        y = sss.sss_gemv(qt, x)
        ref = x.double() @ sss.sss_dequantize(qt).double().T
        assert ((y - ref).abs().amax(1) / ref.abs().amax(1)).max().item() <= TOL
