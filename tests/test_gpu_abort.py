"""A GEMM that gives up while its copies and MMAs are in flight must outlast them: they write shared and tensor
memory that belongs to the next CTA once this one has ended.

A call is held at its start (workspace words 2 and 3); then one copy from the host opens the gate and sets the
status word, as another CTA's timeout would, so the producers issue their stages while every other role gives up, or
the gate opens first and the status follows while the kernel runs.  The next call of the stream, on a workspace of
its own, must compute what it computes alone, bit for bit."""
import time

import numpy as np
import pytest
import torch

from gpu_util import DEV, to_dev_bf16
from paper_2608_26581_gb300 import rfq
from paper_2608_26581_gb300.synth import ActSpec, make_activation, make_weight

pytestmark = pytest.mark.gpu
F4, F8, H, MMA = rfq.RFQ_FMT_MXFP4, rfq.RFQ_FMT_MXFP8, rfq.RFQ_FMT_HIF4, rfq.RFQ_SCALE_MMA
LIMIT_US = 200000


def _abort_then_compute(launch, y, workspace):
    launch(workspace())
    torch.cuda.synchronize()
    want = y.clone()
    assert not torch.isnan(want.float()).any()
    side = torch.cuda.Stream()
    both = torch.tensor([1, LIMIT_US, 1, 1], dtype=torch.int32).pin_memory()   # status, limit, held, gate
    gate = torch.tensor([0, LIMIT_US, 1, 1], dtype=torch.int32).pin_memory()
    for i in range(16):
        ws, ws2 = workspace(), workspace()
        ws[1], ws[2] = LIMIT_US, 1
        y.fill_(float("nan"))
        torch.cuda.synchronize()
        launch(ws)
        launch(ws2)
        time.sleep(0.0005 * (i % 3))
        with torch.cuda.stream(side):
            if i % 2:
                ws[:4].copy_(gate, non_blocking=True)
            ws[:4].copy_(both, non_blocking=True)
        torch.cuda.synchronize()
        assert rfq.rfq_workspace_status(ws) == rfq.RFQ_ERR_TIMEOUT
        assert rfq.rfq_workspace_status(ws2) == rfq.RFQ_OK
        assert torch.equal(y, want), i


def _ws():
    return torch.zeros(rfq.rfq_linear_workspace_bytes() // 4, dtype=torch.int32, device=DEV)


def _x(M, K, seed):
    return to_dev_bf16(make_activation(ActSpec(M, K, "normal", chan_count=2, chan_scale=64.0, seed=seed)))


def _mxfp4(M, K, N, res_fmt=F4):
    wq, xq, xr = rfq.empty_qtensor(F4, MMA, N, K), rfq.empty_qtensor(F4, MMA, M, K), rfq.empty_qtensor(res_fmt, MMA, M, K)
    rfq.rfq_quantize_weight(to_dev_bf16(make_weight(K, N, seed=N)), wq)
    rfq.rfq_quantize_act(_x(M, K, M), xq, xr)
    return wq, xq, xr, torch.empty(M, N, device=DEV)


def _hif4(M, K, N):
    wq, w16 = rfq.empty_qtensor(H, MMA, N, K), rfq.empty_bf16_operand(N, K)
    xq, xr = rfq.empty_qtensor(H, MMA, M, K), rfq.empty_qtensor(H, MMA, M, K)
    xo, ro = rfq.empty_bf16_operand(M, K), rfq.empty_bf16_operand(M, K)
    rfq.rfq_quantize_weight(to_dev_bf16(make_weight(K, N, seed=N)), wq)
    rfq.rfq_dequant(wq, w16.codes)
    rfq.rfq_quantize_act_expand(_x(M, K, M), xq, xr, xo, ro)
    return w16, xq, xr, xo, ro, torch.empty(M, N, device=DEV)


# one CTA per tile, a joint X~ / X^ tile on clusters, X on the M side; fewer stages per CTA than its ring holds
# (the producers end at once) and more
@pytest.mark.parametrize("M,K,N", [(16, 512, 4096), (48, 2048, 4096), (48, 12288, 1024), (333, 1024, 4096),
                                   (333, 6272, 2064)])
def test_cluster_split(M, K, N):
    wq, xq, xr, y = _mxfp4(M, K, N)
    _abort_then_compute(lambda ws: rfq.rfq_linear(xq, xr, None, 256, wq, y, rfq.RFQ_OUT_F32, ws), y, _ws)


@pytest.mark.parametrize("M,K,N", [(32, 1024, 4096), (333, 512, 4096)])
def test_cluster_split_bf16(M, K, N):
    w16, _, _, xo, ro, y = _hif4(M, K, N)
    _abort_then_compute(lambda ws: rfq.rfq_linear(xo, ro, None, 256, w16, y, rfq.RFQ_OUT_F32, ws), y, _ws)


@pytest.mark.parametrize("M", [8, 100])
def test_cluster_split_fused(M):
    K, N = 2048, 4096
    wq = rfq.empty_qtensor(F4, MMA, N, K)
    rfq.rfq_quantize_weight(to_dev_bf16(make_weight(K, N, seed=N)), wq)
    x, y = _x(M, K, M), torch.empty(M, N, device=DEV)
    _abort_then_compute(lambda ws: rfq.rfq_linear_fused(x, wq, y, rfq.RFQ_OUT_F32, ws), y,
                        lambda: rfq.fused_workspace(M, K))


# ---- CTA pairs: both CTAs' copies complete on the even CTA's barriers

@pytest.mark.parametrize("M,K,N", [(600, 640, 15360), (5000, 1024, 2048)])
@pytest.mark.parametrize("tau", [None, 100.0])
def test_pair(M, K, N, tau):
    wq, xq, xr, y = _mxfp4(M, K, N)
    phi = None
    if tau is not None:
        phi = torch.empty(-(-M // 128) * -(-K // 256), dtype=torch.uint8, device=DEV)
        rfq.rfq_quantize_act(_x(M, K, M), xq, xr, phi, mode=rfq.RFQ_FALLBACK_AMAX, tau=tau)
    _abort_then_compute(lambda ws: rfq.rfq_linear(xq, xr, phi, 256, wq, y, rfq.RFQ_OUT_F32, ws), y, _ws)


def test_pair_mixed_rate():
    M, K, N = 700, 512, 528
    wq, xq, xr, y = _mxfp4(M, K, N, res_fmt=F8)
    _abort_then_compute(lambda ws: rfq.rfq_linear_mixed(xq, xr, None, 256, wq, y, rfq.RFQ_OUT_F32, ws), y, _ws)


def test_pair_e4m3():
    M, K, N = 700, 512, 528
    wq, x4, xr, y = _mxfp4(M, K, N, res_fmt=F8)
    x8 = rfq.empty_qtensor(F8, MMA, M, K)
    rfq.rfq_convert(x4, x8)
    _abort_then_compute(lambda ws: rfq.rfq_linear(x8, xr, None, 256, wq, y, rfq.RFQ_OUT_F32, ws), y, _ws)


def test_pair_fused():
    M, K, N = 700, 1024, 1040
    wq = rfq.empty_qtensor(F4, MMA, N, K)
    rfq.rfq_quantize_weight(to_dev_bf16(make_weight(K, N, seed=N)), wq)
    x, y = _x(M, K, M), torch.empty(M, N, device=DEV)
    _abort_then_compute(lambda ws: rfq.rfq_linear_fused(x, wq, y, rfq.RFQ_OUT_F32, ws), y,
                        lambda: rfq.fused_workspace(M, K))


# ---- single CTAs

@pytest.mark.parametrize("counts", [[128, 384, 256], [2176, 2560]])   # (the second on CTA pairs)
def test_grouped(counts):
    K, N, M, G = 1024, 512, sum(counts), len(counts)
    wq, xq, xr = rfq.empty_qtensor(F4, MMA, G * N, K), rfq.empty_qtensor(F4, MMA, M, K), rfq.empty_qtensor(F4, MMA, M, K)
    rfq.rfq_quantize_weight(to_dev_bf16(np.concatenate([make_weight(K, N, seed=g) for g in range(G)], axis=1)), wq)
    rfq.rfq_quantize_act(_x(M, K, M), xq, xr)
    off = torch.from_numpy(np.cumsum([0] + counts).astype(np.int32)).to(DEV)
    y = torch.empty(M, N, device=DEV)
    _abort_then_compute(
        lambda ws: rfq.rfq_linear_grouped(xq, xr, None, 256, off, wq, N, y, rfq.RFQ_OUT_F32, ws), y, _ws)


@pytest.mark.parametrize("codes", [True, False])   # HiF4 expanded inside the GEMM; bf16 operands on whole tiles
def test_hif4_tiled(codes):
    M, K, N = 4096, 256, 4096
    w16, xq, xr, xo, ro, y = _hif4(M, K, N)
    a, r = (xq, xr) if codes else (xo, ro)
    _abort_then_compute(lambda ws: rfq.rfq_linear(a, r, None, 256, w16, y, rfq.RFQ_OUT_F32, ws), y, _ws)
