"""The cluster-split GEMM in each of its forms: every cluster size, W~ or X on the MMA's 128-row side, X~ and X^
joint or apart, every tile width, one or two CTAs per SM.  Each case names the launch shape it is there for and
asserts that the plan search still gives it that one; N ends inside a tile."""
import pytest
import torch

from gpu_util import DEV, check_y, to_dev_bf16
from paper_2608_26581_gb300 import rfq
from paper_2608_26581_gb300.synth import ActSpec, make_activation, make_weight

pytestmark = pytest.mark.gpu
F4, H, B16, MMA = rfq.RFQ_FMT_MXFP4, rfq.RFQ_FMT_HIF4, rfq.RFQ_FMT_BF16, rfq.RFQ_SCALE_MMA

# operands, M, K, N, residual, (cluster, x_on_m, joint, ctas_per_sm, cols)
CASES = [
    (F4, 406, 1920, 8544, 0, (1, 0, 0, 1, 256)), (F4, 259, 128, 8016, 0, (1, 0, 0, 2, 128)),
    (F4, 65, 128, 16, 0, (1, 1, 0, 1, 96)), (F4, 136, 128, 7472, 1, (1, 1, 0, 1, 112)),
    (F4, 267, 128, 6512, 1, (1, 1, 0, 1, 144)), (F4, 264, 128, 7232, 1, (1, 1, 0, 1, 160)),
    (F4, 258, 384, 8304, 0, (1, 1, 0, 1, 176)), (F4, 274, 512, 8864, 1, (1, 1, 0, 1, 192)),
    (F4, 396, 896, 7552, 1, (1, 1, 0, 1, 208)), (F4, 392, 1280, 8464, 0, (1, 1, 0, 1, 224)),
    (F4, 139, 4480, 8624, 0, (2, 0, 0, 1, 256)), (F4, 172, 1408, 6256, 1, (2, 1, 0, 1, 176)),
    (F4, 133, 1920, 7568, 1, (2, 1, 0, 1, 208)), (F4, 1316, 2816, 944, 1, (3, 0, 0, 1, 256)),
    (F4, 1, 3584, 6192, 0, (3, 0, 0, 2, 128)), (F4, 40, 3712, 9296, 1, (3, 0, 1, 1, 256)),
    (F4, 1, 2176, 6352, 1, (3, 0, 1, 2, 128)), (F4, 103, 2176, 6768, 1, (3, 1, 0, 1, 160)),
    (F4, 131, 2176, 5120, 1, (3, 1, 0, 1, 224)), (F4, 1, 2944, 8784, 0, (4, 0, 0, 1, 256)),
    (F4, 1, 4096, 4656, 1, (4, 0, 1, 2, 128)), (F4, 66, 5120, 6784, 0, (4, 1, 0, 1, 192)),
    (F4, 1, 7040, 5696, 1, (6, 0, 1, 1, 256)), (F4, 191, 10368, 1808, 1, (6, 1, 0, 1, 176)),
    (F4, 117, 9344, 16, 1, (8, 1, 0, 1, 96)), (F4, 1418, 7808, 128, 1, (8, 0, 0, 1, 128)),
    (B16, 257, 64, 7712, 0, (1, 0, 0, 2, 128)), (B16, 257, 128, 8256, 0, (1, 1, 0, 1, 176)),
    (B16, 545, 192, 6064, 1, (1, 1, 0, 1, 208)), (B16, 130, 640, 8768, 1, (2, 0, 0, 1, 256)),
    (B16, 1, 896, 5984, 1, (3, 0, 1, 2, 128)), (B16, 285, 960, 3344, 1, (3, 1, 0, 1, 224)),
    (B16, 65, 1216, 6144, 1, (4, 1, 0, 1, 176)), (B16, 1, 1920, 5328, 1, (6, 0, 1, 1, 256)),
    (B16, 18, 6592, 16, 0, (8, 0, 0, 1, 128)), (B16, 1, 5824, 2352, 1, (8, 0, 1, 2, 128)),
    (B16, 344, 4480, 928, 1, (8, 1, 0, 1, 192)),
]


@pytest.mark.parametrize("fmt,M,K,N,res,form", CASES)
def test_form(fmt, M, K, N, res, form):
    plan = rfq.rfq_linear_choice(M, N, K, fmt, bool(res), kernel=rfq.RFQ_KERNEL_CLUSTER)
    assert form == tuple(plan[k] for k in ("cluster", "x_on_m", "joint", "ctas_per_sm", "cols"))
    x = to_dev_bf16(make_activation(ActSpec(M, K, "normal", chan_count=2, chan_scale=64.0, seed=M)))
    qf = F4 if fmt == F4 else H
    q = [rfq.empty_qtensor(qf, MMA, r, K) for r in (N, M, M)]
    op = [rfq.empty_bf16_operand(r, K) for r in (N, M, M)]          # the exact values
    rfq.rfq_quantize_weight(to_dev_bf16(make_weight(K, N, seed=N)), q[0])
    rfq.rfq_quantize_act(x, q[1], q[2] if res else None,
                         mode=rfq.RFQ_FALLBACK_ALL if res else rfq.RFQ_FALLBACK_NONE)
    for t, o in zip(q[:2 + res], op):
        rfq.rfq_dequant(t, o.codes)
    w, xv, rv = (o.codes.double() for o in op)
    a = q if fmt == F4 else op
    y = torch.full((M + 1, N), float("nan"), device=DEV)            # one guard row past Y
    ws = torch.zeros(rfq.rfq_linear_workspace_bytes() // 4, dtype=torch.int32, device=DEV)
    rfq.rfq_linear_on(rfq.RFQ_KERNEL_CLUSTER, a[1], a[2] if res else None, None, 256, a[0], y[:M], rfq.RFQ_OUT_F32, ws)
    assert rfq.rfq_workspace_status(ws) == rfq.RFQ_OK and bool(torch.isnan(y[M]).all())
    check_y(y[:M].double().cpu().numpy(), ((xv + rv if res else xv) @ w.t()).cpu().numpy())


def test_debug_build_checks_the_stores(tmp_path, monkeypatch):
    """The debug build's bounds checks on this kernel's ragged stores."""
    import test_gpu_debug_build as dbg
    cases = dbg._CASES.replace("rfq.rfq_linear(xq", "rfq.rfq_linear_on(rfq.RFQ_KERNEL_CLUSTER, xq")
    fused = "\nyf = torch.zeros(100, N, device='cuda')\n" \
            "rfq.rfq_linear_fused(x[:100].contiguous(), wq, yf, rfq.RFQ_OUT_F32, rfq.fused_workspace(100, K)); keep(yf)\n"
    assert "RFQ_KERNEL_CLUSTER" in cases and "# grouped" in cases
    monkeypatch.setattr(dbg, "_CASES", cases.replace("# grouped", fused + "# grouped"))
    dbg.test_debug_build_records_no_out_of_range_store_and_matches(tmp_path)
