"""rfq_linear_choice and rfq_linear_on on the host: what they refuse, and that every launch shape holds."""
import random

import pytest

from paper_2608_26581_gb300 import _build, rfq

F4, B16 = rfq.RFQ_FMT_MXFP4, rfq.RFQ_FMT_BF16


@pytest.fixture(scope="module", autouse=True)
def lib():
    _build.build()
    return rfq.load_library()


def test_refusals():
    for args, status in (((0, 16, 128), rfq.RFQ_ERR_SHAPE), ((1, 24, 128), rfq.RFQ_ERR_SHAPE),
                         ((1, 16, 192), rfq.RFQ_ERR_SHAPE), ((1, 16, 96, B16), rfq.RFQ_ERR_SHAPE),
                         ((1, 16, 128, 9), rfq.RFQ_ERR_INVALID_ARG),
                         ((1, 16, 128, B16, True, False, True), rfq.RFQ_ERR_INVALID_ARG)):
        with pytest.raises(rfq.RFQError) as e:
            rfq.rfq_linear_choice(*args)
        assert e.value.status == status
    for fmt in (rfq.RFQ_FMT_MXFP8, rfq.RFQ_FMT_HIF4):
        assert rfq.rfq_linear_choice(64, 256, 1024, fmt)["kernel"] == rfq.RFQ_KERNEL_TILED
        with pytest.raises(rfq.RFQError) as e:
            rfq.rfq_linear_choice(64, 256, 1024, fmt, kernel=rfq.RFQ_KERNEL_CLUSTER)
        assert e.value.status == rfq.RFQ_ERR_UNSUPPORTED
    assert rfq.load_library().rfq_linear_on(7, *[None] * 3, 256, *[None] * 2, 0, None, None) == rfq.RFQ_ERR_INVALID_ARG


@pytest.mark.parametrize("fmt", [F4, B16])
def test_every_layer_has_a_launch_shape(fmt):
    rng = random.Random(fmt)
    for _ in range(3000):
        M, N = max(1, int(2 ** rng.uniform(0, 15))), 16 * max(1, int(2 ** rng.uniform(0, 11)))
        K = (128 if fmt == F4 else 64) * max(1, int(2 ** rng.uniform(0, 8)))
        for res in (False, True):
            p = rfq.rfq_linear_choice(M, N, K, fmt, res, kernel=rfq.RFQ_KERNEL_CLUSTER)
            stages_k = -(-K // (256 if fmt == F4 else 64))
            assert 1 <= p["cluster"] <= min(8, stages_k) and p["stages"] >= 2
            assert p["rows"] % 16 == 0 and 16 <= p["rows"] <= 128 and p["cols"] % 16 == 0 and p["cols"] <= 256
            # the chosen kernel is one of the two, and a cluster choice is the plan above
            a = rfq.rfq_linear_choice(M, N, K, fmt, res)
            assert a["kernel"] == rfq.RFQ_KERNEL_TILED or a == p


T, C = rfq.RFQ_KERNEL_TILED, rfq.RFQ_KERNEL_CLUSTER


# layers timed on both kernels (quantizer + GEMM, us), apart by a tenth or more
@pytest.mark.parametrize("fmt,M,K,N,kernel", [
    (F4, 2500, 13824, 5120, T),    # 77 on the tiled kernel, 124 on the cluster-split one
    (F4, 1777, 12288, 4096, T),    # 48, 74
    (F4, 1000, 8192, 8192, T),     # 34, 46
    (F4, 512, 5120, 13824, T),     # 24, 33
    (F4, 16, 4096, 24576, T),      # 15.8, 19.9 (GEMM)
    (F4, 128, 12288, 4096, C),     # 28, 14 (GEMM)
    (F4, 256, 12288, 4096, C),     # 24, 19 (GEMM)
    (B16, 64, 3584, 18944, T),     # 36, 51
    (B16, 1777, 4096, 4096, T),    # 61, 83
    (B16, 256, 13824, 5120, C),    # 93, 39 (GEMM)
    (B16, 64, 8192, 8192, C),      # 59, 46 (GEMM)
])
def test_choice_without_a_residual(fmt, M, K, N, kernel):
    assert rfq.rfq_linear_choice(M, N, K, fmt, residual=False)["kernel"] == kernel


# with phi 0 on every tile, where the tiled kernels do least
@pytest.mark.parametrize("fmt,M,K,N,kernel", [
    (F4, 1000, 13824, 5120, T),    # 55, 71
    (F4, 400, 13824, 5120, T),     # 33, 38
    (F4, 128, 12288, 4096, C),     # 37, 17
    (F4, 256, 12288, 4096, C),     # 33, 23
    (B16, 333, 5120, 13824, T),    # 82, 96
    (B16, 300, 5120, 13824, T),    # 82, 95
    (B16, 256, 12288, 4096, C),    # 96, 44
])
def test_choice_with_phi(fmt, M, K, N, kernel):
    assert rfq.rfq_linear_choice(M, N, K, fmt, phi=True)["kernel"] == kernel


@pytest.mark.parametrize("M,K,N,kernel", [(32, 3584, 18944, T),     # 43.5, 48.5
                                          (32, 12288, 4096, C)])    # 111, 22 (GEMM)
def test_choice_bf16_decode(M, K, N, kernel):
    assert rfq.rfq_linear_choice(M, N, K, B16)["kernel"] == kernel


# 128 rows quantized inside the GEMM: 96 tiles in one wave of single CTAs take 40.6 us, in three waves of clusters of
# four 59.8
def test_fused_wide_layer_is_one_wave():
    assert rfq.rfq_linear_choice(128, 24576, 4096, residual=False, fused=True)["cluster"] == 1
