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


@pytest.mark.parametrize("batch", [2, 9])
@pytest.mark.parametrize("q", [2, 4])
@pytest.mark.parametrize("n,k,g,grid", [
    (24, 32, 32, sss.GRID_ASYM),            # one group: a quarter of a step
    (65, 96, 32, sss.GRID_SIGNED_SYM),      # 2-byte scale rows, q = 2 code rows of 8 bytes' alignment
    (40, 192, 64, sss.GRID_ASYM),           # a step and a half
    (33, 128, 128, sss.GRID_SIGNED_SYM),    # one step, one scale per row
    (100, 4128, 32, sss.GRID_ASYM),         # a quarter of a step past 32
    (2500, 1120, 32, sss.GRID_UNSIGNED_SYM),
    (300, 4224, 128, sss.GRID_ASYM),        # 66-byte scale rows
    (70, 4160, 64, sss.GRID_SIGNED_SYM),
])
def test_gemv_cluster_cut_steps(n, k, g, grid, q, batch):
    run_case(n, k, q, g, grid, batch, n + k + g + q + batch, outliers=False, tol=TOL)


@pytest.mark.parametrize("q", [2, 4])
def test_gemv_cluster_cut_steps_with_stale_memory(q):
    # what other launches left in shared memory (all bits set: NaN as scales)
    # has no part in a cut step
    w = inputs.student_t_weights_cuda(64, 1024, 11, outliers=False)
    full = sss.sss_quantize(w, q, 32, sss.GRID_ASYM)
    full.codes.fill_(255)
    full.scales.fill_(-1)
    full.mins.fill_(-1)
    cut = sss.sss_quantize(w[:, :864].contiguous(), q, 32, sss.GRID_ASYM)
    x = inputs.normal_bf16_cuda((16, 1024), 12)
    xc = x[:, :864].contiguous()
    ref = xc.double() @ sss.sss_dequantize(cut).double().T
    for _ in range(20):
        sss.sss_gemv(full, x)
        y = sss.sss_gemv(cut, xc)
        assert ((y - ref).abs().amax(1) / ref.abs().amax(1)).max().item() <= TOL


@pytest.mark.parametrize("k", [512, 544])  # whole steps, and a last one cut short
@pytest.mark.parametrize("q,grid", [(4, sss.GRID_SIGNED_SYM), (2, sss.GRID_UNSIGNED_SYM), (4, sss.GRID_ASYM)])
@pytest.mark.parametrize("mag", [1e-8, 1e-6, 1e-5, 1e-4])
def test_gemv_cluster_small_activations(mag, q, grid, k):
    # below 2^-13 the operand fl16(x 2^-p) holds x rounded; the product has to be
    # that of the rounded values, symmetric offset and minimum included
    qt = sss.sss_quantize(inputs.student_t_weights_cuda(100, k, 13, outliers=False), q, 32, grid)
    x = (inputs.normal_bf16_cuda((5, k), 14).float() * mag).bfloat16()
    pos = torch.tensor([0., 4., 0., 4.] if q == 4 else [2., 0., 2., 0.], device="cuda")
    p2 = torch.exp2(pos.repeat(k // 4))  # of elements e and e + 4 of every eight
    held = (x.float() / p2).half().double() * p2.double()
    w = sss.sss_dequantize(qt).double()
    # an output is a chain of at most 40 fp32 or tensor-core additions, each off by
    # 2^-23 of the magnitudes that it adds: codes are up to 2^q <= 16 steps, so a
    # term is up to 16 max|w| |x|
    bound = 40 * 2.0**-23 * (held.abs().sum(1, keepdim=True) * 16 * w.abs().amax(1))
    assert ((sss.sss_gemv(qt, x) - held @ w.T).abs() <= bound).all()


@pytest.mark.parametrize("n,k", [(100, 1024), (300, 4352), (70, 544)])
@pytest.mark.parametrize("q,grid", [(4, sss.GRID_SIGNED_SYM), (2, sss.GRID_SIGNED_SYM),
                                    (2, sss.GRID_ASYM), (4, sss.GRID_ASYM)])
def test_gemv_cluster_activations_beyond_fp16(q, grid, n, k):
    qt = sss.sss_quantize(inputs.student_t_weights_cuda(n, k, 15, outliers=False), q, 32, grid)
    x = inputs.normal_bf16_cuda((16, k), 16)
    plain = sss.sss_gemv(qt, x)
    x[1] *= 65536.0           # many from 65520 on
    x[2, 5] = 1e30            # one, of any size
    x[7, k - 1] = float("inf")
    x[9, 0] = float("-inf")
    x[15, 3] = float("nan")
    y = sss.sss_gemv(qt, x)
    ref = x.double() @ sss.sss_dequantize(qt).double().T
    same = [b for b in range(16) if b not in (1, 2, 7, 9, 15)]
    assert torch.equal(y[same], plain[same])
    for b in (1, 2):
        assert ((y[b] - ref[b]).abs().max() / ref[b].abs().max()).item() <= TOL
    for b in (7, 9, 15):  # +-inf by the weight's sign, NaN where it is zero
        assert torch.equal(y[b].isnan(), ref[b].isnan())
        assert torch.equal(y[b].nan_to_num(0.0), ref[b].float().nan_to_num(0.0))


@pytest.mark.parametrize("batch", [3, 16])
@pytest.mark.parametrize("n,k,g,grid", [
    (200, 1024, 32, sss.GRID_SIGNED_SYM), (200, 1024, 128, sss.GRID_UNSIGNED_SYM),
    (2048, 2048, 64, sss.GRID_SIGNED_SYM), (600, 1056, 32, sss.GRID_SIGNED_SYM),
])
def test_gemv_cluster_q2_symmetric_is_exact_products(n, k, g, grid, batch):
    # fp32 sums of exact products: of the order of the square root of the chain's
    # length, up to 64 additions here, times 2^-24
    qt = sss.sss_quantize(inputs.student_t_weights_cuda(n, k, 17, outliers=False), 2, g, grid)
    x = inputs.normal_bf16_cuda((batch, k), 18)
    ref = x.double() @ sss.sss_dequantize(qt).double().T
    assert ((sss.sss_gemv(qt, x) - ref).norm() / ref.norm()).item() <= 8 * 2.0**-24


@pytest.mark.parametrize("q,grid,g,batch,k", [
    (4, sss.GRID_ASYM, 32, 16, 12288), (4, sss.GRID_ASYM, 64, 9, 12288),
    (4, sss.GRID_SIGNED_SYM, 32, 16, 16384), (4, sss.GRID_SIGNED_SYM, 128, 9, 21504),
    (2, sss.GRID_ASYM, 32, 16, 22528), (2, sss.GRID_SIGNED_SYM, 128, 9, 28672),
    (4, sss.GRID_ASYM, 32, 8, 30720), (4, sss.GRID_SIGNED_SYM, 64, 2, 45056),
])
def test_gemv_cluster_longest_rows(q, grid, g, batch, k):
    # the longest k whose staged activations fit a cluster: fp32 sums; and the next
    # multiple of 256, the batched kernel: weights rounded to fp16
    for kk, tol in ((k, TOL), (k + 256, 2.0**-11)):
        qt = sss.sss_quantize(inputs.student_t_weights_cuda(40, kk, 19, outliers=False), q, g, grid)
        x = inputs.normal_bf16_cuda((batch, kk), 20)
        y = sss.sss_gemv(qt, x)
        ref = x.double() @ sss.sss_dequantize(qt).double().T
        err = ((y - ref).abs().amax(1) / ref.abs().amax(1)).max().item()
        assert err <= tol
        if tol != TOL and q == 4:  # (symmetric weights at q = 2 are exact in fp16)
            assert err > TOL
