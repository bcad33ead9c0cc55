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
