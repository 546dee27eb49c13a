"""Many rows by few output columns: layers of more than 1024 rows that the cluster-split GEMM takes, and their
neighbours that stay with the tiled kernels, against the fp64 oracle."""
import pytest
import torch

from gpu_util import DEV, check_y, qtensor_host, to_dev_bf16
from paper_2608_26581_gb300 import rfq
from paper_2608_26581_gb300.synth import ActSpec, make_activation, make_weight

pytestmark = pytest.mark.gpu
F4, H, MMA = rfq.RFQ_FMT_MXFP4, rfq.RFQ_FMT_HIF4, rfq.RFQ_SCALE_MMA


def _inputs(M, K, N):
    xb = make_activation(ActSpec(M, K, "normal", chan_count=2, chan_scale=64.0, tok_count=1, tok_scale=50.0, seed=M))
    return to_dev_bf16(xb), to_dev_bf16(make_weight(K, N, seed=N))


# row tiles that end one row past a tile and that divide evenly, clusters of 1 to 8, ragged columns, the last
# shape of a full wave of 256 x 256 tiles and the first beyond it
@pytest.mark.parametrize("M,K,N", [(1025, 2176, 528), (1300, 4096, 16), (2049, 1152, 800), (4096, 2048, 512),
                                   (19456, 256, 256), (19457, 256, 256)])
@pytest.mark.parametrize("mode", [rfq.RFQ_FALLBACK_ALL, rfq.RFQ_FALLBACK_AMAX])
def test_mxfp4(orc, M, K, N, mode):
    if mode == rfq.RFQ_FALLBACK_AMAX and K % 256:
        pytest.skip("whole 256-column tiles here")
    x, w = _inputs(M, K, N)
    wq, xq, xr = (rfq.empty_qtensor(F4, MMA, r, K) for r in (N, M, M))
    phi = torch.empty(-(-M // 128) * -(-K // 256), dtype=torch.uint8, device=DEV)
    rfq.rfq_quantize_weight(w, wq)
    rfq.rfq_quantize_act(x, xq, xr, phi, mode=mode, tau=100.0)
    y = torch.full((M + 1, N), float("nan"), device=DEV)   # one guard row past Y
    ws = torch.zeros(rfq.rfq_linear_workspace_bytes() // 4, dtype=torch.int32, device=DEV)
    rfq.rfq_linear(xq, xr, phi if mode == rfq.RFQ_FALLBACK_AMAX else None, 256, wq, y[:M], rfq.RFQ_OUT_F32, ws)
    assert rfq.rfq_workspace_status(ws) == rfq.RFQ_OK and bool(torch.isnan(y[M]).all())
    # (the stored residual of a phi = 0 tile is zero)
    check_y(y[:M].double().cpu().numpy(),
            orc.linear(orc.FMT_MXFP4, *qtensor_host(xq), *qtensor_host(xr), *qtensor_host(wq), M, K, N))


@pytest.mark.parametrize("M,K,N", [(1025, 1088, 528), (1300, 2048, 16), (2049, 576, 800), (4096, 1024, 512)])
def test_hif4(orc, M, K, N):
    x, w = _inputs(M, K, N)
    row = rfq.RFQ_SCALE_ROWMAJOR
    wq, xq, xr = (rfq.empty_qtensor(H, row, r, K) for r in (N, M, M))
    w16, xo, ro = (rfq.empty_bf16_operand(r, K) for r in (N, M, M))
    rfq.rfq_quantize_weight(w, wq)
    rfq.rfq_dequant(wq, w16.codes)
    rfq.rfq_quantize_act_expand(x, xq, xr, xo, ro)
    y = torch.full((M + 1, N), 7.0, dtype=torch.bfloat16, device=DEV)
    ws = torch.zeros(rfq.rfq_linear_workspace_bytes() // 4, dtype=torch.int32, device=DEV)
    rfq.rfq_linear(xo, ro, None, 256, w16, y[:M], rfq.RFQ_OUT_BF16, ws)
    assert rfq.rfq_workspace_status(ws) == rfq.RFQ_OK and bool((y[M] == 7.0).all())
    check_y(y[:M].double().cpu().numpy(),
            orc.linear(orc.FMT_HIF4, *qtensor_host(xq), *qtensor_host(xr), *qtensor_host(wq), M, K, N), bf16=True)


# between one and three waves of the tiled kernels' tiles (taken: 80 and 96 tiles for 76 pairs, 180 for 152 CTAs)
# and beyond three, against an fp64 product of the same operand values
@pytest.mark.parametrize("fmt,M,K,N", [(F4, 1025, 4096, 4096), (F4, 1800, 1024, 2560), (F4, 5000, 384, 3600),
                                       (H, 1025, 4096, 5120), (H, 2600, 4096, 2048), (H, 5000, 320, 3088)])
def test_waves(fmt, M, K, N):
    x, w = _inputs(M, K, N)
    lay = MMA if fmt == F4 else rfq.RFQ_SCALE_ROWMAJOR
    q = [rfq.empty_qtensor(fmt, lay, r, K) for r in (N, M, M)]
    op = [rfq.empty_bf16_operand(r, K) for r in (N, M, M)]   # the exact values
    rfq.rfq_quantize_weight(w, q[0])
    rfq.rfq_quantize_act(x, q[1], q[2])
    val = []
    for t, o in zip(q, op):
        rfq.rfq_dequant(t, o.codes)
        val.append(o.codes.view(torch.bfloat16).view(t.rows, K).double())
    y = torch.full((M + 1, N), float("nan"), device=DEV)
    ws = torch.zeros(rfq.rfq_linear_workspace_bytes() // 4, dtype=torch.int32, device=DEV)
    a = q if fmt == F4 else op
    rfq.rfq_linear(a[1], a[2], None, 256, a[0], y[:M], rfq.RFQ_OUT_F32, ws)
    assert rfq.rfq_workspace_status(ws) == rfq.RFQ_OK and bool(torch.isnan(y[M]).all())
    check_y(y[:M].double().cpu().numpy(), ((val[1] + val[2]) @ val[0].t()).cpu().numpy())
