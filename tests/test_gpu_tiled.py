"""The tiled GEMM kernels by name.  rfq_linear chooses between them and the cluster-split kernel by estimated time, so
which kernel a test of rfq_linear runs is not the test's to say: here the tests of the tiled kernels' epilogues, phi
records and bounded waits run with that choice taken away (rfq_linear_on)."""
import functools

import pytest
import torch

import test_gpu_abort as _abort
import test_gpu_debug_build as _debug
from paper_2608_26581_gb300 import rfq
from test_gpu_hif4 import (test_linear_no_residual_and_phi, test_linear_shapes,  # noqa: F401
                           test_phi_records_wrap)
from test_gpu_linear import (test_bf16_output, test_phi_amax_many_stage_blocks, test_phi_amax_records_wrap,  # noqa: F401
                             test_phi_amax_skips_residual_tiles, test_phi_beyond_record_capacity_falls_back_exactly,
                             test_plain_w4a4_without_residual, test_ragged_shapes, test_repeated_calls_are_deterministic)
from test_gpu_timeout import test_hif4_gemm_timeout, test_mxfp4_gemm_timeout  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def tiled(monkeypatch):
    monkeypatch.setattr(rfq, "rfq_linear", functools.partial(rfq.rfq_linear_on, rfq.RFQ_KERNEL_TILED))


# in flight when the call gives up: one CTA per tile, CTA pairs with fewer stages than their ring holds and with more
@pytest.mark.parametrize("M,K,N", [(100, 512, 1040), (600, 512, 528), (600, 2176, 528)])
def test_abort_mxfp4(M, K, N):
    _abort.test_cluster_split(M, K, N)


@pytest.mark.parametrize("M,K,N", [(32, 1024, 4096), (333, 128, 1040)])
def test_abort_bf16(M, K, N):
    _abort.test_cluster_split_bf16(M, K, N)


def test_debug_build_checks_the_pair_epilogue(tmp_path, monkeypatch):
    """The debug build's bounds checks on the CTA-pair kernel's ragged stores, its operands quantized beforehand."""
    monkeypatch.setattr(_debug, "_CASES", _debug._CASES.replace("rfq.rfq_linear(xq", "rfq.rfq_linear_on(rfq.RFQ_KERNEL_TILED, xq"))
    assert "RFQ_KERNEL_TILED" in _debug._CASES
    _debug.test_debug_build_records_no_out_of_range_store_and_matches(tmp_path)


def test_rows_sum_alike_in_calls_of_every_size():
    """A row's Y has the same bits whether its call has 700 rows or 1 (single CTAs up to 128 rows, pairs beyond)."""
    M, K, N = 700, 4224, 1040
    wq, xq, xr, y = _abort._mxfp4(M, K, N)
    x = _abort._x(M, K, M)
    rfq.rfq_linear(xq, xr, None, 256, wq, y, rfq.RFQ_OUT_F32, _abort._ws())
    for a, b in ((0, 1), (128, 256), (384, 700), (699, 700)):
        q, r = (rfq.empty_qtensor(rfq.RFQ_FMT_MXFP4, rfq.RFQ_SCALE_MMA, b - a, K) for _ in range(2))
        rfq.rfq_quantize_act(x[a:b].contiguous(), q, r)
        part = torch.empty(b - a, N, device="cuda")
        rfq.rfq_linear(q, r, None, 256, wq, part, rfq.RFQ_OUT_F32, _abort._ws())
        assert torch.equal(part, y[a:b]), (a, b)
