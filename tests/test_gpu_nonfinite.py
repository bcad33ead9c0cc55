"""Quantizers of tensors that hold NaN and infinities (needs a B200): what becomes of those elements, of their block's scale and of
the block's other elements, on every kernel.  Codes and scales are compared byte for byte."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_28358_b200 import inputs, mq
from parity_util import dev, host

pytestmark = pytest.mark.gpu

# N, C, H, W: positions that are a multiple of four (small, at most 16 rows, whole lines), and that are none (staged runs, items of 8 and 16)
SHAPES = {"aligned": (40, 48, 8, 8), "rows16": (12, 40, 8, 8), "lines": (64, 64, 36, 36), "few": (300, 700, 3, 3), "odd8": (40, 48, 5, 7), "odd16": (300, 200, 7, 9)}
NAN_CODE = {mq.E4M3: 0x7F, mq.E5M2: 0x7F, mq.E2M1: 7, mq.E3M2: 0x1F, mq.E2M3: 0x1F}      # formats without a NaN: the largest magnitude
PATTERNS = np.array([0x7FC00000, 0x7FFFFFFF, 0xFFC00001, 0x7F800001], np.uint32)          # quiet, all ones, negative, signalling


def tensor(name, specials, share=0.002):
    rng = np.random.default_rng(7)
    x = rng.standard_normal(SHAPES[name]).astype(np.float32)
    at = rng.random(x.shape) < share
    x.view(np.uint32)[at] = rng.choice(specials, int(at.sum()))
    n, c, h, w = x.shape
    return inputs.ConvDesc(n, c, h, w, 32, 1, 1, 1, 1, 0, 0), x


def logical(q, x, fmt):
    """The stored codes [position][N][C rounded up to 32] as an array like x."""
    n, c, h, w = x.shape
    codes = host(q.codes)
    if fmt == mq.E2M1:
        codes = np.stack([codes & 15, codes >> 4], -1).reshape(-1)
    return codes.reshape(h * w, n, -1)[:, :, :c].transpose(1, 2, 0).reshape(x.shape)


def source(x, layout):
    return dev(x if layout == mq.NCHW else np.ascontiguousarray(x.transpose(2, 3, 0, 1)))


@pytest.mark.parametrize("layout", [mq.NCHW, mq.HWNC], ids=["nchw", "hwnc"])
@pytest.mark.parametrize("fmt", sorted(NAN_CODE))
@pytest.mark.parametrize("name", SHAPES)
def test_nan_elements(name, fmt, layout):
    """Both roundings make the same code of a NaN, and of an infinity the largest magnitude with its sign."""
    d, x = tensor(name, np.concatenate([PATTERNS, np.array([np.inf, -np.inf], np.float32).view(np.uint32)]))
    sign = {mq.E2M1: 8, mq.E3M2: 0x20, mq.E2M3: 0x20}.get(fmt, 0x80)
    top = {mq.E4M3: 0x7E, mq.E5M2: 0x7B, mq.E2M1: 7}.get(fmt, 0x1F)
    for block in (mq.TILE32, mq.LINE32):
        for q in (mq.quantize(d, mq.ROLE_X, fmt, source(x, layout), src_layout=layout, block=block),
                  mq.quantize_sr(d, mq.ROLE_X, fmt, source(x, layout), 5, src_layout=layout, block=block)):
            codes = logical(q, x, fmt)
            assert (codes[np.isnan(x)] == NAN_CODE[fmt]).all(), np.unique(codes[np.isnan(x)])
            assert (codes[np.isposinf(x)] == top).all() and (codes[np.isneginf(x)] == top | sign).all()
    assert mq.last_device_status() == 0


@pytest.mark.parametrize("seed", [None, 5], ids=["nearest", "stochastic"])
@pytest.mark.parametrize("layout", [mq.NCHW, mq.HWNC], ids=["nchw", "hwnc"])
@pytest.mark.parametrize("name", SHAPES)
def test_paper_format(name, layout, seed):
    """Eq. 6 of a NaN, in a block that is not zero, is the largest magnitude; in a block that encodes to zeros, as with T_scale 0 or
    infinite, it and an infinity are zeros with their sign.  The other elements are the oracle's."""
    b16 = (16, 16)
    amax = lambda v: torch.tensor([v], dtype=torch.float32, device="cuda")
    d, x = tensor(name, PATTERNS)
    q = mq.quantize_ts(d, mq.ROLE_X, source(x, layout), src_layout=layout, amax_in=amax(3.0), seed=seed)
    codes, scales = oracle.quantize_ts(d, mq.ROLE_X, np.nan_to_num(x, nan=0.0), b16, amax=3.0, seed=seed)[:2]
    want = logical(mq.QTensor(torch.from_numpy(codes), None, mq.E2M1, mq.ROLE_X), x, mq.E2M1)
    assert np.array_equal(host(q.scales), scales) and host(q.tensor_scale)[1] == np.nanmax(np.abs(x))
    assert np.array_equal(logical(q, x, mq.E2M1), np.where(np.isnan(x), 7, want))
    d, x = tensor(name, np.concatenate([PATTERNS, np.array([np.inf, -np.inf], np.float32).view(np.uint32)]))
    sign = np.where(np.signbit(x), 8, 0)
    for am in (None, 0.0, np.inf, np.nan):        # None: the tensor's own maximum, which is infinite
        q = mq.quantize_ts(d, mq.ROLE_X, source(x, layout), src_layout=layout, amax_in=None if am is None else amax(am), seed=seed)
        assert np.array_equal(logical(q, x, mq.E2M1), sign), am
    q = mq.quantize_ts(d, mq.ROLE_X, source(x, layout), src_layout=layout, amax_in=amax(3.0), seed=seed)
    got = logical(q, x, mq.E2M1)
    assert (got[np.isnan(x)] == 7).all() and (got[np.isinf(x)] == 7 + sign[np.isinf(x)]).all()


@pytest.mark.parametrize("fmt", sorted(NAN_CODE))
@pytest.mark.parametrize("name", SHAPES)
def test_scales_of_blocks_with_a_nan(name, fmt):
    """Where the positions are no multiple of four, and in small tensors of line blocks, a block with a NaN has the scale of an infinite maximum, under which its finite
    elements are zeros with their sign; elsewhere the maximum passes over the NaN.  All other bytes are the oracle's."""
    d, x = tensor(name, PATTERNS, 0.0005)
    n, c, h, w = x.shape
    infinite = min(255 - {mq.E4M3: 8, mq.E5M2: 15, mq.E3M2: 4}.get(fmt, 2), 254)
    sign = {mq.E2M1: 8, mq.E3M2: 0x20, mq.E2M3: 0x20}.get(fmt, 0x80)
    for block, side in ((mq.TILE32, 32), (mq.LINE32, 1)):
        codes, scales = oracle.quantize(d, mq.ROLE_X, fmt, np.nan_to_num(x, nan=0.0), (side, 32))
        want = logical(mq.QTensor(torch.from_numpy(codes), None, fmt, mq.ROLE_X), x, fmt)
        scales = scales.reshape(h * w, (n + side - 1) // side, -1)
        if (h * w) % 4 != 0 or (block == mq.LINE32 and x.size < 1 << 18):
            rows, chans, ys, xs = np.nonzero(np.isnan(x))
            marked = np.zeros(scales.shape, bool)
            marked[ys * w + xs, rows // side, chans // 32] = True
            scales = np.where(marked, infinite, scales)
            of = np.repeat(np.repeat(marked, side, 1)[:, :n], 32, 2)[:, :, :c].transpose(1, 2, 0).reshape(x.shape)
            want = np.where(of, np.where(np.signbit(x), sign, 0), want)
        want = np.where(np.isnan(x), NAN_CODE[fmt], want)
        q = mq.quantize(d, mq.ROLE_X, fmt, source(x, mq.NCHW), block=block)
        assert np.array_equal(host(q.scales), scales.reshape(-1))
        assert np.array_equal(logical(q, x, fmt), want)
