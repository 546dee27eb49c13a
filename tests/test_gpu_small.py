"""The few-rows GEMM (X on the narrow MMA side, the reduction split over a
cluster) against the fp64 oracle: edges of its row tiles, odd 128-element
chunk counts, ragged output columns, every operand kind, and the order of its
sums (the same Y on every run and for row chunks of a matrix)."""
import numpy as np
import pytest
import torch

from gpu_util import DEV, check_y, qtensor_host, to_dev_bf16
from paper_2608_26581_gb300 import rfq
from paper_2608_26581_gb300.synth import ActSpec, make_activation, make_weight

pytestmark = pytest.mark.gpu
F4, H, MMA = rfq.RFQ_FMT_MXFP4, rfq.RFQ_FMT_HIF4, rfq.RFQ_SCALE_MMA


def _ws():
    return torch.zeros(rfq.rfq_linear_workspace_bytes() // 4, dtype=torch.int32, device=DEV)


def _xw(M, K, N, seed):
    xb = make_activation(ActSpec(M, K, "normal", chan_count=2, chan_scale=64.0, tok_count=1, tok_scale=50.0, seed=seed))
    return xb, make_weight(K, N, seed=seed + 1)


# rows around the 16-row granule, the 64-row limit of the joint X~ / X^ tile and the 128-row tile; reductions
# of 1 to 48 stages (split over clusters of 1 to 8); N ends inside a 16-column group's, a 128-row block's and a tile's
@pytest.mark.parametrize("M,K,N", [(1, 128, 16), (1, 4096, 528), (15, 384, 48), (16, 2176, 272), (17, 1024, 144),
                                   (33, 12288, 400), (48, 640, 1552), (64, 2048, 1536), (65, 2048, 1536),
                                   (80, 3968, 1008), (100, 4096, 4112), (127, 896, 1296), (128, 8192, 640),
                                   (129, 2048, 1536), (200, 4096, 2064), (333, 6272, 1040), (500, 2304, 1552),
                                   (900, 2048, 1520)])
@pytest.mark.parametrize("res,out", [(True, rfq.RFQ_OUT_F32), (False, rfq.RFQ_OUT_BF16)])
def test_mxfp4(orc, M, K, N, res, out):
    xb, wb = _xw(M, K, N, seed=M + K)
    wq, xq = rfq.empty_qtensor(F4, MMA, N, K), rfq.empty_qtensor(F4, MMA, M, K)
    xr = rfq.empty_qtensor(F4, MMA, M, K) if res else None
    rfq.rfq_quantize_weight(to_dev_bf16(wb), wq)
    rfq.rfq_quantize_act(to_dev_bf16(xb), xq, xr, mode=rfq.RFQ_FALLBACK_ALL if res else rfq.RFQ_FALLBACK_NONE)
    dt = torch.float32 if out == rfq.RFQ_OUT_F32 else torch.bfloat16
    buf = torch.full((M + 1, N), 7.0, dtype=dt, device=DEV)   # one guard row past Y
    y, ws = buf[:M], _ws()
    rfq.rfq_linear(xq, xr, None, 256, wq, y, out, ws)
    again = torch.empty(M, N, dtype=dt, device=DEV)
    rfq.rfq_linear(xq, xr, None, 256, wq, again, out, ws)
    assert rfq.rfq_workspace_status(ws) == rfq.RFQ_OK
    assert torch.equal(y, again) and bool((buf[M] == 7.0).all())
    mc, ms = qtensor_host(xq)
    rc, rs = qtensor_host(xr) if res else (None, None)
    wc, wsf = qtensor_host(wq)
    check_y(y.double().cpu().numpy(), orc.linear(orc.FMT_MXFP4, mc, ms, rc, rs, wc, wsf, M, K, N),
            bf16=out == rfq.RFQ_OUT_BF16)


@pytest.mark.parametrize("M,K,N", [(1, 128, 16), (8, 4096, 1040), (16, 384, 272), (17, 2048, 1536), (60, 1152, 144),
                                   (64, 640, 400), (65, 2048, 528), (128, 4096, 640)])
@pytest.mark.parametrize("mode", [rfq.RFQ_FALLBACK_ALL, rfq.RFQ_FALLBACK_NONE])
def test_fused(orc, M, K, N, mode):
    xb, wb = _xw(M, K, N, seed=M + N)
    wq = rfq.empty_qtensor(F4, MMA, N, K)
    rfq.rfq_quantize_weight(to_dev_bf16(wb), wq)
    y = torch.full((M, N), float("nan"), device=DEV)
    ws = rfq.fused_workspace(M, K, mode)
    rfq.rfq_linear_fused(to_dev_bf16(xb), wq, y, rfq.RFQ_OUT_F32, ws, mode=mode)
    assert rfq.rfq_workspace_status(ws) == rfq.RFQ_OK
    res = mode == rfq.RFQ_FALLBACK_ALL
    q = orc.quantize_act(xb, orc.FMT_MXFP4, orc.PHI_ALL if res else orc.PHI_NONE)
    wc, wsf = orc.quantize_weight(wb)
    check_y(y.double().cpu().numpy(), orc.linear(orc.FMT_MXFP4, q["main_codes"], q["main_scales"], q["res_codes"],
                                                 q["res_scales"], wc, wsf, M, K, N))


@pytest.mark.parametrize("M,K,N", [(1, 64, 16), (16, 4096, 272), (33, 12288, 400), (64, 1088, 1536), (65, 2048, 1552),
                                   (128, 4032, 144), (129, 2048, 1536), (333, 4096, 1040), (700, 2048, 1520)])
@pytest.mark.parametrize("res", [True, False])
def test_hif4(orc, M, K, N, res):
    xb, wb = _xw(M, K, N, seed=M + K + N)
    wq = rfq.empty_qtensor(H, rfq.RFQ_SCALE_ROWMAJOR, N, K)
    rfq.rfq_quantize_weight(to_dev_bf16(wb), wq)
    w16 = rfq.empty_bf16_operand(N, K)
    rfq.rfq_dequant(wq, w16.codes)
    xq, xo = rfq.empty_qtensor(H, rfq.RFQ_SCALE_ROWMAJOR, M, K), rfq.empty_bf16_operand(M, K)
    xr = rfq.empty_qtensor(H, rfq.RFQ_SCALE_ROWMAJOR, M, K) if res else None
    ro = rfq.empty_bf16_operand(M, K) if res else None
    rfq.rfq_quantize_act_expand(to_dev_bf16(xb), xq, xr, xo, ro,
                                mode=rfq.RFQ_FALLBACK_ALL if res else rfq.RFQ_FALLBACK_NONE)
    y, ws = torch.full((M, N), float("nan"), device=DEV), _ws()
    rfq.rfq_linear(xo, ro, None, 256, w16, y, rfq.RFQ_OUT_F32, ws)
    assert rfq.rfq_workspace_status(ws) == rfq.RFQ_OK
    mc, ms = qtensor_host(xq)
    rc, rs = qtensor_host(xr) if res else (None, None)
    wc, wsf = qtensor_host(wq)
    check_y(y.double().cpu().numpy(), orc.linear(orc.FMT_HIF4, mc, ms, rc, rs, wc, wsf, M, K, N))


def test_row_chunks_sum_as_the_whole():
    """Host chunks of 128 rows, the last of them two rows, against one call on the whole matrix: bit for bit."""
    M, K, N = 258, 4096, 1040
    xb, wb = _xw(M, K, N, seed=9)
    wq = rfq.empty_qtensor(F4, MMA, N, K)
    rfq.rfq_quantize_weight(to_dev_bf16(wb), wq)
    xq, xr = rfq.empty_qtensor(F4, MMA, M, K), rfq.empty_qtensor(F4, MMA, M, K)
    x, y, yd = to_dev_bf16(xb), torch.empty(M, N, device=DEV), torch.empty(M, N, device=DEV)
    rfq.rfq_quantize_act(x, xq, xr)
    rfq.rfq_linear(xq, xr, None, 256, wq, y, rfq.RFQ_OUT_F32, _ws())
    yh = torch.empty(M, N)
    rfq.rfq_linear_host(torch.from_numpy(xb.view(np.int16)).view(torch.bfloat16), wq, yh, rfq.RFQ_OUT_F32,
                        torch.empty_like(x), xq, xr, None, yd, _ws(), chunk_rows=128)
    torch.cuda.synchronize()
    assert torch.equal(yh, y.cpu())
