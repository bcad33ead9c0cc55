"""The paper-format quantizer's element rounding where it is decided without a division (needs a B200): values at and a few units in
the last place around every decision threshold, denominators that are powers of two, others, and so extreme that every
element is divided; tensors with few positions (staged runs), and maxima by the cluster reduction around its largest size.
Codes, scales and the recorded maximum are the oracle's bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_28358_b200 import inputs, mq
from parity_util import assert_same_bytes, dev, host

pytestmark = pytest.mark.gpu

B16 = (16, 16)


def check(name, d, role, x, amax=None, seed=None, layout=mq.NCHW):
    o = oracle.quantize_ts(d, role, x, B16, amax=None if amax is None else float(amax), seed=seed)
    src = x if layout == mq.NCHW else np.ascontiguousarray(x.transpose(0, 2, 3, 1) if role == mq.ROLE_W else x.transpose(2, 3, 0, 1))
    a = None if amax is None else torch.tensor([amax], dtype=torch.float32, device="cuda")
    g = mq.quantize_ts(d, role, dev(src), src_layout=layout, amax_in=a, seed=seed)
    assert_same_bytes(g.scales, o[1], f"{name} block scales")
    assert_same_bytes(g.codes, o[0], f"{name} codes")
    st = host(g.tensor_scale)
    assert st[1] == np.abs(x).max() and st[0] == np.float32(o[2]), (name, st, o[2])


@pytest.mark.parametrize("scale", [1.0, 0.7310585, 3e-34, 1e34], ids=["pow2", "odd", "tiny", "huge"])
@pytest.mark.parametrize("route", ["lines", "blocks", "hwnc"])
def test_around_thresholds(knobs, scale, route):
    """Every 16 x 16 block holds its maximum 6 den and, in its other places, thresholds of both roundings times den, moved by up
    to six units in the last place."""
    knobs(MQ_QUANT_TMA=1 if route == "lines" else 0)
    d = inputs.conv_desc(32, 32, 8, 8, 32, 1, 1, 0)
    rng = np.random.default_rng(3)
    marks = np.array([0.25, 0.5, 0.75, 1.0, 1.25, 1.5, 1.75, 2.0, 2.5, 3.0, 3.5, 4.0, 5.0, 5.5, 6.0, 0.0, 0.1])
    x = (rng.choice(marks, (32, 32, 8, 8)) * scale).astype(np.float32)
    x = (x.view(np.int32) + np.where(x == 0, 0, rng.integers(-6, 7, x.shape)).astype(np.int32)).view(np.float32)
    x *= rng.choice(np.float32([-1.0, 1.0]), x.shape)
    x[::16, ::16] = np.float32(6.0 * scale)
    amax = np.float32(448.0) * np.float32(6.0) * np.float32(scale) / np.float32(256.0)     # T_scale = scale / 256, Scale_b = 256
    layout = mq.HWNC if route == "hwnc" else mq.NCHW
    check(f"{route} {scale}", d, mq.ROLE_X, x, amax, None, layout)
    check(f"{route} {scale} own maximum", d, mq.ROLE_X, x, None, None, layout)
    check(f"{route} {scale} stochastic", d, mq.ROLE_X, x, amax, 17, layout)


@pytest.mark.parametrize("seed", [None, 5])
@pytest.mark.parametrize("shape", [(3, 40, 50, 1), (70, 37, 3, 3), (33, 35, 5, 5), (17, 16, 3, 13), (16, 48, 6, 7)], ids=str)
def test_few_positions(shape, seed):
    """Weight-like tensors [C_out][C_in][Kh][Kw]: one tap, 3x3, 5x5, the most positions the staged runs take (39), and one more
    than that (42); ragged rows and channels; the first also as an activation of more than 2^17 elements."""
    co, ci, kh, kw = shape
    d = inputs.ConvDesc(2, ci, kh + 1, kw + 1, co, kh, kw, 1, 1, 0, 0)
    w = np.random.default_rng(9).standard_normal((co, ci, kh, kw)).astype(np.float32)
    w[0, :, 0, 0] = 0.0
    check(f"W {shape}", d, mq.ROLE_W, w, None, seed)
    check(f"W {shape} supplied", d, mq.ROLE_W, w, np.float32(2.0), seed)
    d = inputs.ConvDesc(300, 64, 3, 3, 32, 1, 1, 1, 1, 0, 0)
    check("X 3x3", d, mq.ROLE_X, inputs.make_x(d, 2, "gauss"), np.float32(3.0), seed)


@pytest.mark.parametrize("n", [(1, 2), (32, 1024), (33, 1024)], ids=str)
def test_own_maximum_reduction(n):
    """One pixel; 2^20 elements, the cluster reduction's most, and just above (the last element is the largest)."""
    rows, c = n
    d = inputs.ConvDesc(rows, c, 4, 8, 32, 1, 1, 1, 1, 0, 0)
    x = np.random.default_rng(rows).standard_normal((rows, c, 4, 8)).astype(np.float32)
    x[-1, -1, -1, -1] = -37.5
    check(f"max of {x.size}", d, mq.ROLE_X, x)
