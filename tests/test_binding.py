"""The binding's native marshalling (_mq_torch): argument errors, and - on a GPU - caller-owned outputs, workspaces and streams,
alone and from several threads at once."""
from concurrent.futures import ThreadPoolExecutor

import pytest
import torch

from paper_2609_28358_b200 import inputs, mq

D = inputs.conv_desc(40, 48, 6, 7, 70, 3, 1, 1)


class _NullStream:
    cuda_stream = 0


def _small(role):
    return mq.QTensor(torch.zeros(8, dtype=torch.uint8), torch.zeros(8, dtype=torch.uint8), mq.E4M3, role)


def test_argument_errors_are_python_exceptions():
    with pytest.raises(AssertionError):
        mq.quantize(D, mq.ROLE_X, mq.E4M3, torch.zeros(40, 48, 6, 7))          # not a CUDA tensor
    with pytest.raises(TypeError):
        mq.quantize(D[:5], mq.ROLE_X, mq.E4M3, torch.zeros(40, 48, 6, 7))
    with pytest.raises(AttributeError):
        mq.conv_fwd(D, 3, 4)
    for call in (lambda: mq.conv_fwd(D, _small(mq.ROLE_X), _small(mq.ROLE_W), stream=_NullStream()), lambda: mq.cbf_im2col(D, _small(mq.ROLE_X), stream=_NullStream()),
                 lambda: mq.conv_fwd_mx(D, _small(mq.ROLE_X), _small(mq.ROLE_W), mq.E4M3, stream=_NullStream())):
        with pytest.raises(mq.MqError) as e:                                    # refused on the host, nothing launched
            call()
        assert e.value.status == 4
    with pytest.raises(KeyError):
        mq.conv_fwd(D, _small(mq.ROLE_X), _small(mq.ROLE_W), dtype=torch.float16, stream=_NullStream())


def test_arguments_are_taken_as_they_were_through_ctypes():
    q = _small(mq.ROLE_X), _small(mq.ROLE_W)
    call = lambda d=D, **kw: mq.conv_fwd(d, *q, stream=_NullStream(), **kw)
    for bad in (dict(layout=0.0), dict(layout="0")):                            # neither floats nor text are integers
        with pytest.raises(TypeError):
            call(**bad)
    with pytest.raises(TypeError):
        mq.conv_fwd(D, mq.QTensor(q[0].codes, q[0].scales, 0.0, mq.ROLE_X), q[1], stream=_NullStream())
    for good in (dict(dtype=None), dict(layout=True), dict(d=[float(v) for v in D])):   # PyTorch's default type; int()'s arguments as extents
        with pytest.raises(mq.MqError) as e:
            call(**good)
        assert e.value.status == 4


def _pass(x, w, dy, **kw):
    qs = [mq.quantize(D, r, mq.E4M3, t, **kw) for r, t in enumerate((x, w, dy))]
    return [mq.conv_fwd(D, qs[0], qs[1], **kw), mq.conv_bwd_data(D, qs[1], qs[2], **kw), mq.conv_bwd_weight(D, qs[0], qs[2], **kw)]


@pytest.mark.gpu
def test_caller_owned_buffers_streams_and_threads():
    x, w, dy = [torch.from_numpy(f(D, 5)).cuda() for f in (inputs.make_x, inputs.make_w, inputs.make_dy)]
    want = _pass(x, w, dy)
    torch.cuda.synchronize()
    # outputs and workspace of the caller's: written in place and returned
    q = mq.empty_qtensor(D, mq.ROLE_X, mq.E4M3)
    assert mq.quantize(D, mq.ROLE_X, mq.E4M3, x, out=q) is q
    wq = mq.quantize(D, mq.ROLE_W, mq.E4M3, w)
    y = torch.full_like(want[0], float("nan"))
    ws = torch.empty(mq.workspace_size(D, mq.OP_FWD, mq.E4M3, mq.E4M3), dtype=torch.uint8, device="cuda")
    assert mq.conv_fwd(D, q, wq, y=y, workspace=ws).data_ptr() == y.data_ptr()
    torch.cuda.synchronize()
    assert torch.equal(y, want[0])
    with pytest.raises(mq.MqError):
        mq.conv_bwd_weight(D, q, mq.quantize(D, mq.ROLE_DY, mq.E4M3, dy), workspace=ws[:16])

    # each thread on a stream of its own
    def work(i):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            got = [_pass(x, w, dy, stream=s if i % 2 else None) for _ in range(20)][-1]
        s.synchronize()
        return all(torch.equal(a, b) for a, b in zip(got, want))

    with ThreadPoolExecutor(4) as ex:
        assert all(ex.map(work, range(8)))
    assert mq.last_device_status() == 0


@pytest.mark.gpu
def test_a_stream_that_is_not_the_current_one():
    """Calls given a stream while another is current: neither stream's work reaches memory that the other still uses."""
    d = inputs.conv_desc(64, 128, 28, 28, 128, 3, 1, 1)
    x, x2, w, dy = [torch.from_numpy(f(d, s)).cuda() for f, s in ((inputs.make_x, 5), (inputs.make_x, 6), (inputs.make_w, 5), (inputs.make_dy, 5))]
    qs = [mq.quantize(d, r, mq.E4M3, t) for r, t in enumerate((x, w, dy))]
    q2 = mq.quantize(d, mq.ROLE_X, mq.E4M3, x2)
    calls = [lambda **kw: mq.conv_fwd(d, qs[0], qs[1], **kw), lambda **kw: mq.conv_bwd_data(d, qs[1], qs[2], **kw), lambda **kw: mq.conv_bwd_weight(d, qs[0], qs[2], **kw),
             lambda **kw: mq.conv_fwd_mx(d, qs[0], qs[1], mq.E4M3, **kw).codes, lambda **kw: mq.quantize(d, mq.ROLE_X, mq.E4M3, x, **kw).codes,
             lambda **kw: mq.cbf_im2col(d, qs[0], **kw)[0], lambda **kw: mq.conv_bwd_data_static(d, qs[1], qs[2], **kw)]
    ops = [(mq.OP_FWD, 0, 0), (mq.OP_BWD_DATA, 0, 0), (mq.OP_BWD_WEIGHT, 0, 0)]
    sizes = [mq.workspace_size(d, *o) for o in ops] + [mq.conv_mx_workspace_size(d, mq.OP_FWD, 0, 0)]
    want = [c() for c in calls]
    want2 = mq.conv_fwd(d, q2, qs[1])
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for call, ref in zip(calls, want):
        nbytes = sizes + [ref.numel() * ref.element_size()]
        # the current stream is about to overwrite blocks of the call's sizes that were dropped just before the call
        torch.cuda._sleep(20_000_000)
        for n in nbytes:
            torch.empty(n, dtype=torch.uint8, device="cuda").fill_(0xA5)
        got = call(stream=side)
        side.synchronize()
        torch.cuda.synchronize()
        assert torch.equal(got, ref)
        # ... and blocks given out right after it, before its kernels have started
        with torch.cuda.stream(side):
            torch.cuda._sleep(20_000_000)
        got = call(stream=side)
        for n in nbytes:
            torch.empty(n, dtype=torch.uint8, device="cuda").fill_(0xA5)
        torch.cuda.synchronize()
        assert torch.equal(got, ref)
    # a result read on the current stream and dropped while that read is waiting
    y = mq.conv_fwd(d, qs[0], qs[1], stream=side)
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda._sleep(20_000_000)
    z = y + 0.0
    del y
    y2 = mq.conv_fwd(d, q2, qs[1], stream=side)
    torch.cuda.synchronize()
    assert torch.equal(z, want[0]) and torch.equal(y2, want2)
    assert mq.last_device_status() == 0
