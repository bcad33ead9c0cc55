"""Strides of eight and more (needs a B200), as in patch embeddings: the copy engine steps over at most eight columns, so the
forward GEMM and the weight gradient of wider strides run on the CUDA-core kernels.  Against the CPU oracle."""
import pytest
import torch

import oracle
from paper_2609_28358_b200 import inputs, mq
from parity_util import GEMM_TOL, OracleLayer, assert_gemm_close, check_convs, check_quantize, dev
from test_gpu_fused_epilogue import check_emitted

pytestmark = pytest.mark.gpu

# N, C_in, H, W, C_out, kernel = stride, padding
SHAPES = [(5, 3, 32, 40, 48, 8, 8, 0), (5, 3, 27, 36, 48, 9, 9, 0), (3, 64, 32, 48, 40, 16, 16, 0)]


@pytest.mark.parametrize("fmts", [(mq.E2M1,) * 3, (mq.E4M3, mq.E4M3, mq.E5M2), (mq.E3M2_P6, mq.E4M3, mq.E5M2)], ids=["fp4", "fp8", "packed6"])
@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_gemms(shape, fmts):
    d = inputs.conv_desc(*shape)
    base = tuple(mq.E3M2 if f == mq.E3M2_P6 else f for f in fmts)
    ol = OracleLayer(inputs.Layer("wide stride", d, *base, "relu", "kaiming", "gauss", 3))
    qs = check_quantize(ol)
    if fmts != base:
        qs[0] = mq.quantize(d, mq.ROLE_X, fmts[0], dev(ol.src[0]))
    check_convs(ol, qs, layouts=(mq.NCHW, mq.HWNC))
    if fmts == base:
        y64, ab = oracle.conv_fwd(d, *ol.hat[:2])
        ho, wo = inputs.out_hw(d)
        yq = mq.conv_fwd_mx(d, qs[0], qs[1], fmts[0], mq.ACT_RELU)
        check_emitted("wide stride", d._replace(C_in=d.C_out, H=ho, W=wo), oracle.ROLE_X, fmts[0], y64, GEMM_TOL * ab, mq.ACT_RELU, yq)
    assert mq.last_device_status() == 0


@pytest.mark.parametrize("block", [mq.LINE32, mq.TS16], ids=["line", "ts16"])
@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_forward_of_other_blocks(shape, block):
    d = inputs.conv_desc(*shape)
    roles, src = (mq.ROLE_X, mq.ROLE_W), (inputs.make_x(d, 4, "gauss"), inputs.make_w(d, 4))
    if block == mq.TS16:
        q = [mq.quantize_ts(d, r, dev(t)) for r, t in zip(roles, src)]
        hat = [oracle.dequant_ts(d, r, *oracle.quantize_ts(d, r, t, (16, 16))[:3], (16, 16)) for r, t in zip(roles, src)]
        assert mq.conv_fwd_ts(d, q[0], q[1], torch.tensor([4.0], device="cuda")).codes.numel() > 0
    else:
        q = [mq.quantize(d, r, mq.E2M1, dev(t), block=block) for r, t in zip(roles, src)]
        hat = [oracle.dequant(d, r, mq.E2M1, *oracle.quantize(d, r, mq.E2M1, t, (1, 32)), (1, 32)) for r, t in zip(roles, src)]
    ref, ab = oracle.conv_fwd(d, *hat)
    assert_gemm_close(mq.conv_fwd(d, q[0], q[1]), ref, ab, "forward")
    assert mq.last_device_status() == 0
