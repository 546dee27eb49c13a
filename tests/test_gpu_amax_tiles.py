"""The AMAX quantizer's two block sizes: a matrix with more 128 x 256 tiles than the 16-warp form takes, against the
same rows quantized in pieces that it takes (which test_gpu_quant compares with the oracle).  Whole numbers: equal."""
import pytest
import torch

from gpu_util import DEV
from paper_2608_26581_gb300 import rfq

pytestmark = pytest.mark.gpu


def _quantize(x, layout):
    M, K = x.shape
    xq, xr = rfq.empty_qtensor(rfq.RFQ_FMT_MXFP4, layout, M, K), rfq.empty_qtensor(rfq.RFQ_FMT_MXFP4, layout, M, K)
    phi = torch.empty(-(-M // 128) * (K // 256), dtype=torch.uint8, device=DEV)
    rfq.rfq_quantize_act(x, xq, xr, phi, mode=rfq.RFQ_FALLBACK_AMAX, tau=200.0)
    return [xq.codes, xq.scales, xr.codes, xr.scales, phi]


@pytest.mark.parametrize("layout", [rfq.RFQ_SCALE_MMA, rfq.RFQ_SCALE_ROWMAJOR])
@pytest.mark.parametrize("blocks", [0, 1])   # tiles: the 16-warp form's last, the 8-warp form's first
def test_pieces_equal_the_whole(layout, blocks):
    rows, K = 128 * (8 * torch.cuda.get_device_properties(0).multi_processor_count + blocks), 512
    M = rows - 37
    g = torch.Generator(device=DEV)
    g.manual_seed(5)
    x = torch.empty(M, K, dtype=torch.bfloat16, device=DEV).normal_(0.0, 1.0, generator=g)
    x[torch.randperm(M, generator=g, device=DEV)[:64]] *= 200.0
    whole = _quantize(x, layout)
    cut = 128 * (rows // 256)
    parts = zip(_quantize(x[:cut], layout), _quantize(x[cut:], layout))
    assert 0 < int(whole[4].sum()) < whole[4].numel()
    for w, (a, b) in zip(whole, parts):
        assert torch.equal(w, torch.cat([a, b]))
