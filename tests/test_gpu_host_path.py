"""The host-buffer path beside other work: callers on streams of their own, and a layer that changes streams."""

import pytest
import torch

import paper_2512_02541_b200 as P
from paper_2512_02541_b200 import inputs

from test_gpu_parity import _cfgs

pytestmark = pytest.mark.gpu

WL = inputs.Workload("host_path", 6, 12, 13, 5, 4, 64, 4, 1, 2, "proj")


def _case(seed):
    """Pinned Q, K, V and an output buffer, and the output of the resident forward (and every kernel of either path loaded: the
    first launch of one waits for the device)."""
    Q, K, V = inputs.make_qkv(WL, seed=seed, device="cuda")
    layer = P.SubsampledGlobalAttention(_cfgs(WL)[0])
    want = layer.forward(Q, K, V).cpu()
    host = [t.cpu().pin_memory() for t in (Q, K, V)]
    out = torch.empty_like(host[0]).pin_memory()
    layer.forward_host(*host, out)
    torch.cuda.synchronize()
    return host, out.fill_(float("nan")), want


def test_a_caller_does_not_wait_for_another_streams_work():
    (h1, o1, w1), (h2, o2, w2) = _case(1), _case(2)
    first, second = (P.SubsampledGlobalAttention(_cfgs(WL)[0]) for _ in range(2))
    busy, free = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(2):   # a layer's first call, which waits for all of its stream's work, and a later one
        with torch.cuda.stream(busy):
            torch.cuda._sleep(int(1e9))       # about half a second
            first.forward_host(*h1, o1)
        with torch.cuda.stream(free):
            second.forward_host(*h2, o2)
        free.synchronize()
        assert not busy.query(), "the second caller's copies stood behind the first one's work"
        assert torch.equal(o2, w2)
        busy.synchronize()
        assert torch.equal(o1, w1)


def test_a_layer_called_on_one_stream_and_then_on_another():
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    (h1, o1, w1), (h2, o2, w2) = _case(3), _case(4)
    layer = P.SubsampledGlobalAttention(_cfgs(WL)[0])
    torch.cuda.synchronize()
    for _ in range(3):
        b.wait_stream(a)
        a.wait_stream(b)
        with torch.cuda.stream(a):
            layer.forward_host(*h1, o1)
        b.wait_stream(a)
        with torch.cuda.stream(b):
            layer.forward_host(*h2, o2)
        a.wait_stream(b)
    layer.check_status()
    assert torch.equal(o1, w1) and torch.equal(o2, w2)


def test_inputs_that_a_copy_still_writes():
    """Pinned inputs filled by an asynchronous copy on the calling stream, in a second call (a first one waits for the stream)."""
    (h1, o1, w1), (h2, _, w2) = _case(5), _case(6)
    device = [t.cuda() for t in h2]
    layer = P.SubsampledGlobalAttention(_cfgs(WL)[0])
    layer.forward_host(*h1, o1)
    torch.cuda.synchronize()
    assert torch.equal(o1, w1)
    torch.cuda._sleep(int(1e8))       # so that the copies below are far from done when the call is made
    for host, dev in zip(h1, device):
        host.copy_(dev, non_blocking=True)
    written = torch.cuda.Event()
    written.record()
    layer.forward_host(*h1, o1, inputs_ready=written)
    layer.check_status()
    assert torch.equal(o1, w2)
