"""Channel rows that no box of the tensor-core GEMMs divides (needs a B200): rows of 16, 48, 80, 112 and 144 bytes (E2M1), which end
inside an MMA's 32-byte K-atom and are completed by the copy engine's zero fill, and rows of 96, 160 and 224 bytes, whose last
128-byte chunk is short.  Forward, input gradient and quantizing epilogue against the CPU oracle."""
import pytest

import oracle
from paper_2609_28358_b200 import inputs, mq
from parity_util import GEMM_TOL, OracleLayer, assert_gemm_close, check_convs, check_quantize, dev
from test_gpu_fused_epilogue import check_emitted

pytestmark = pytest.mark.gpu

SHAPES = [
    ("rows16_48", (20, 32, 6, 8, 96, 3, 1, 1)),        # one K-atom of which half is padding; whole-tile kernel
    ("rows48_80", (40, 96, 5, 7, 160, 3, 1, 1)),
    ("rows112_144_s2", (33, 224, 7, 8, 288, 3, 2, 1)),  # stride 2: parity classes of the input gradient
    ("rows96_k1", (36, 192, 6, 6, 96, 1, 1, 0)),
    ("rows16_k1", (3, 32, 6, 9, 160, 1, 1, 0)),        # E2M1: sums of 32 products, few of them - on the CUDA cores
    ("rows16_k1_one", (1, 32, 40, 44, 160, 1, 1, 0)),  # ... and the quantizing epilogue of one sample
    ("rows16_k5", (9, 16, 9, 8, 352, 5, 1, 2)),        # three channel tiles on a thin contraction (weight tile reloaded)
]


@pytest.mark.parametrize("fmts", [(mq.E2M1,) * 3, (mq.E4M3, mq.E4M3, mq.E5M2), (mq.E2M3,) * 3], ids=["fp4", "fp8", "fp6"])
@pytest.mark.parametrize("name,shape", SHAPES, ids=[s[0] for s in SHAPES])
def test_gemms(name, shape, fmts):
    d = inputs.conv_desc(*shape)
    ol = OracleLayer(inputs.Layer(name, d, *fmts, "relu", "kaiming", "gauss", 31))
    qs = check_quantize(ol)
    check_convs(ol, qs, layouts=(mq.NCHW, mq.HWNC))
    if fmts[0] != mq.E2M3:
        y64, ab = oracle.conv_fwd(d, *ol.hat[:2])
        ho, wo = inputs.out_hw(d)
        yq = mq.conv_fwd_mx(d, qs[0], qs[1], fmts[0], mq.ACT_RELU)
        check_emitted(name, d._replace(C_in=d.C_out, H=ho, W=wo), oracle.ROLE_X, fmts[0], y64, GEMM_TOL * ab, mq.ACT_RELU, yq)
        assert mq.last_device_status() == 0


@pytest.mark.parametrize("block", [mq.LINE32, mq.TS16], ids=["line", "ts16"])
@pytest.mark.parametrize("name,shape", SHAPES, ids=[s[0] for s in SHAPES])
def test_other_block_shapes(name, shape, block):
    d = inputs.conv_desc(*shape)
    src = (inputs.make_x(d, 32, "relu"), inputs.make_w(d, 32), inputs.make_dy(d, 32, "gauss"))
    roles = (mq.ROLE_X, mq.ROLE_W, mq.ROLE_DY)
    if block == mq.TS16:
        gq = [mq.quantize_ts(d, r, dev(t)) for r, t in zip(roles, src)]
        hat = [oracle.dequant_ts(d, r, *oracle.quantize_ts(d, r, t, (16, 16))[:3], (16, 16)) for r, t in zip(roles, src)]
        ref, ab = oracle.conv_bwd_data(d, hat[1], hat[2])
        assert_gemm_close(mq.conv_bwd_data(d, gq[1], gq[2]), ref, ab, f"{name} bwd_data")
    else:
        gq = [mq.quantize(d, r, mq.E2M1, dev(t), block=block) for r, t in zip(roles[:2], src)]
        hat = [oracle.dequant(d, r, mq.E2M1, *oracle.quantize(d, r, mq.E2M1, t, (1, 32)), (1, 32)) for r, t in zip(roles[:2], src)]
    ref, ab = oracle.conv_fwd(d, hat[0], hat[1])
    assert_gemm_close(mq.conv_fwd(d, gq[0], gq[1]), ref, ab, f"{name} fwd")
    assert mq.last_device_status() == 0
