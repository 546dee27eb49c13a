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
