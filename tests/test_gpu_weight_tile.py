"""The tiled weight quantizer (even N: 128 columns x 256 rows per block) and the
general form (odd N) against the oracle, bytes for bytes: a single pair of
columns, ends inside a tile in both directions, whole tiles."""
import numpy as np
import pytest
import torch

from gpu_util import qtensor_host, to_dev_bf16
from paper_2608_26581_gb300 import rfq
from paper_2608_26581_gb300.synth import make_weight

pytestmark = pytest.mark.gpu
ROW, MMA = rfq.RFQ_SCALE_ROWMAJOR, rfq.RFQ_SCALE_MMA


@pytest.mark.parametrize("fmt,layout,K", [(rfq.RFQ_FMT_MXFP4, ROW, 32), (rfq.RFQ_FMT_MXFP4, ROW, 288),
                                          (rfq.RFQ_FMT_MXFP4, MMA, 128), (rfq.RFQ_FMT_MXFP4, MMA, 640),
                                          (rfq.RFQ_FMT_MXFP8, ROW, 288), (rfq.RFQ_FMT_MXFP8, MMA, 384),
                                          (rfq.RFQ_FMT_HIF4, ROW, 64), (rfq.RFQ_FMT_HIF4, ROW, 320),
                                          (rfq.RFQ_FMT_HIF4, MMA, 576)])
@pytest.mark.parametrize("N", [1, 2, 127, 128, 130, 258])
def test_weight_bytes(orc, fmt, layout, K, N):
    wb = make_weight(K, N, seed=K + N)
    wb[:, 0] = 0                                     # an all-zero column
    wb[K // 2, N - 1] = 0x7F7F                       # the largest bf16
    q = rfq.empty_qtensor(fmt, layout, N, K)
    q.codes.fill_(0xAB)
    q.scales.fill_(0xAB)
    rfq.rfq_quantize_weight(to_dev_bf16(wb), q)
    codes, scales = qtensor_host(q)
    ofmt = {rfq.RFQ_FMT_MXFP4: orc.FMT_MXFP4, rfq.RFQ_FMT_MXFP8: orc.FMT_MXFP8, rfq.RFQ_FMT_HIF4: orc.FMT_HIF4}[fmt]
    rc, rs = orc.quantize_weight(wb, ofmt)
    assert np.array_equal(scales, rs) and np.array_equal(codes, rc)
    if layout == MMA and fmt != rfq.RFQ_FMT_HIF4:    # the padding rows' scale bytes are zero
        sf = q.scales[: -(-N // 128) * 128 * (K // 32)].cpu().numpy().reshape(-1, K // 128, 32, 4, 4)
        rows = np.arange(32)[:, None] + 32 * np.arange(4)[None, :]
        pad = rows >= N - (sf.shape[0] - 1) * 128
        assert not sf[-1][:, pad].any()
