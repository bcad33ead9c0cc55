"""mq_conv_bwd_data_static on layers whose fastest tiles need more scratch than the static array holds: those that smaller scratch
serves are accepted - tiles of the fewest scale chunks, or the CUDA-core kernels for 4-bit rows that end inside an MMA's K-atom -
and give the workspace call's result."""
import ctypes

import pytest
import torch

from paper_2609_28358_b200 import inputs, mq

TS = "ts16"
# N, C_in, H, W, C_out, kernel, stride, padding; formats; scratch of the fastest tiles, MB
CASES = [((40, 26, 65, 65, 517, 5, 3, 2), mq.E4M3, 18.8), ((40, 26, 65, 65, 517, 5, 3, 2), mq.E2M1, 22.2), ((40, 26, 65, 65, 517, 5, 3, 2), TS, 44.2),
         ((52, 96, 55, 55, 160, 7, 2, 3), mq.E4M3, 24.7), ((8, 32, 94, 94, 320, 7, 2, 3), mq.E2M1, 18.9), ((16, 32, 134, 22, 320, 5, 2, 2), TS, 20.0)]
IDS = [f"{c[0][0]}x{c[0][1]}_{c[0][2]}_{c[1]}" for c in CASES]


def _operands(fmt):
    return (mq.E2M1, mq.TS16) if fmt == TS else (fmt, mq.TILE32)


@pytest.mark.parametrize("shape,fmt,mb", CASES, ids=IDS)
def test_accepted(shape, fmt, mb):
    if torch.cuda.is_available():
        pytest.skip("host checks only: the addresses below are no memory")
    d, (f, block) = inputs.conv_desc(*shape), _operands(fmt)
    need = mq.workspace_size(d, mq.OP_BWD_DATA, f, f, block)
    assert need > mq.STATIC_SCRATCH_BYTES and abs(need / 1e6 - mb) < 0.1
    q = [mq._QTensor(4096, 4096, 1 << 40, 1 << 40, f, r, block, 4096) for r in (mq.ROLE_W, mq.ROLE_DY)]
    for layout in (mq.NCHW, mq.HWNC):
        st = mq.lib().mq_conv_bwd_data_static(ctypes.byref(mq._d(d)), ctypes.byref(q[0]), ctypes.byref(q[1]), ctypes.c_void_p(4096), mq.F32, layout, None)
        assert st == 5          # MQ_ERR_CUDA: accepted, and there is no device


@pytest.mark.gpu
@pytest.mark.parametrize("shape,fmt,mb", CASES, ids=IDS)
def test_matches_the_workspace_call(shape, fmt, mb):
    d, (f, block) = inputs.conv_desc(*shape), _operands(fmt)
    w, dy = [torch.from_numpy(t).cuda() for t in (inputs.make_w(d, 3), inputs.make_dy(d, 3, "gauss"))]
    if fmt == TS:
        q = mq.quantize_ts(d, mq.ROLE_W, w), mq.quantize_ts(d, mq.ROLE_DY, dy)
    else:
        q = mq.quantize(d, mq.ROLE_W, f, w), mq.quantize(d, mq.ROLE_DY, f, dy)
    for layout in (mq.NCHW, mq.HWNC):
        want = mq.conv_bwd_data(d, *q, layout=layout).double()
        got = mq.conv_bwd_data_static(d, *q, layout=layout).double()
        # the same products in fp32 sums of another order: 8e-7 apart in the 2-norm at most over the library's layers
        assert (got - want).norm() <= 4e-6 * want.norm()
    assert mq.last_device_status() == 0
