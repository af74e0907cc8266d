"""The Python binding's own work, without a GPU: where the outputs that it allocates come from, and what it refuses."""
import contextlib
import subprocess
import sys
from pathlib import Path

import pytest

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def dq():
    from paper_1904_01197_b200 import build
    build.build()
    import paper_1904_01197_b200 as dq
    return dq


def _calls_that_allocate(dq):
    p = dq.DqParams(512, 2, 3)
    g = torch.zeros(1000)
    m = [dq.Message(torch.zeros(63, dtype=torch.int32), torch.zeros(2), 1, 0, dq.DQ_KIND_DQSG, p)]
    return {
        "dqsg_encode": lambda s: dq.dqsg_encode(g, 1, 0, 0, p, stream=s),
        "ndqsg_encode": lambda s: dq.ndqsg_encode(g, 1, 0, 0, p, stream=s),
        "dqsg_encode_range": lambda s: dq.dqsg_encode_range(g, 512, 1, 0, 0, p, stream=s),
        "ndqsg_encode_range": lambda s: dq.ndqsg_encode_range(g, 512, 1, 0, 0, p, stream=s),
        "dqsg_decode_aggregate": lambda s: dq.dqsg_decode_aggregate(m, 1000, 0, stream=s),
        "ndqsg_decode_aggregate": lambda s: dq.ndqsg_decode_aggregate(m, 1000, 0, None, stream=s),
        "range": lambda s: dq.ndqsg_decode_aggregate_range(m, 1000, 512, 0, None, stream=s),
        "half": lambda s: dq.dqsg_decode_aggregate_half_dithered(m, 1000, stream=s),
        "running": lambda s: dq.ndqsg_decode_aggregate_running(m, 1000, 0, stream=s),
        "first": lambda s: dq.ndqsg_decode_aggregate_side_first(m, 1000, 0, stream=s),
        "histogram": lambda s: dq.code_histogram(m[0].packed, 1000, 2, stream=s),
        "ternary_pack": lambda s: dq.ternary_pack(m[0].packed, 1000, stream=s),
        "ternary_unpack": lambda s: dq.ternary_unpack(torch.zeros(200, dtype=torch.uint8), 1000, stream=s),
    }


class _Stream:
    cuda_stream = 0x1230


class _FakeCalls:
    """In the place of the native calls: every call succeeds without a GPU."""
    encode = decode = code_histogram = ternary_pack = ternary_unpack = staticmethod(lambda *a: 0)


@pytest.mark.parametrize("given", [True, False])
def test_outputs_are_allocated_on_the_stream_of_the_call(dq, monkeypatch, given):
    entered, allocated_in = [], []

    @contextlib.contextmanager
    def on(stream):
        entered.append(stream)
        yield
        entered.pop()

    def new_output(numel, dtype, device):
        allocated_in.append(list(entered))
        return torch.empty(numel, dtype=dtype)

    monkeypatch.setattr(torch.cuda, "stream", on)
    monkeypatch.setattr(torch.cuda, "ExternalStream", lambda ptr, device: ("stream", ptr))
    monkeypatch.setattr(dq.binding, "new_output", new_output)
    monkeypatch.setattr(dq.binding, "_calls_module", _FakeCalls)
    for name, call in _calls_that_allocate(dq).items():
        allocated_in.clear()
        call(_Stream if given else None)
        assert allocated_in, name
        assert all(a == ([("stream", 0x1230)] if given else []) for a in allocated_in), name


def test_an_encode_without_a_gradient_is_refused(dq):
    p = dq.DqParams(512, 2, 3)
    out = torch.zeros(63, dtype=torch.int32), torch.zeros(2)
    for encode in (dq.dqsg_encode, dq.ndqsg_encode):
        with pytest.raises(TypeError, match="grad"):
            encode(None, 1, 0, 0, p, *out, stream=_Stream)
    # the buffers are as necessary as the gradient
    with pytest.raises(TypeError):
        dq.binding._calls().encode(dq.DQ_KIND_DQSG, None, 0, 1, 0, 0, p, None, None, _Stream)


# Tensors under vmap have no storage: torch throws when their address is asked for.
_VMAPPED = """
import sys
sys.path.insert(0, sys.argv[1])
import torch
from torch._subclasses.fake_tensor import FakeTensorMode
import paper_1904_01197_b200 as dq

class Stream:
    cuda_stream = 0

p = dq.DqParams(512, 2, 3)
with FakeTensorMode(allow_non_fake_inputs=True):
    f32, i32, u8 = (torch.empty(3, 1024, dtype=t, device="cuda:0") for t in (torch.float32, torch.int32, torch.uint8))
    pk, sc, out = i32[0], f32[0], f32[1]
    for name, x, call in (
            ("encode", f32, lambda x: dq.dqsg_encode(x, 1, 0, 0, p, pk, sc, stream=Stream)),
            ("decode", i32, lambda x: dq.dqsg_decode_aggregate([dq.Message(x, sc, 1, 0, 0, p)], 1024, 0, out, stream=Stream)),
            ("histogram", i32, lambda x: dq.code_histogram(x, 1024, 2, torch.empty(4, dtype=torch.int64, device="cuda:0"),
                                                           stream=Stream)),
            ("pack", i32, lambda x: dq.ternary_pack(x, 1024, u8[0], stream=Stream)),
            ("unpack", u8, lambda x: dq.ternary_unpack(x, 1024, pk, stream=Stream))):
        def body(t):
            try:
                call(t)
            except RuntimeError as e:
                print(name, "raised", "storage" in str(e))
            return t
        torch.vmap(body)(x)
"""


def test_a_tensor_without_storage_raises_and_does_not_end_the_process(dq):
    r = subprocess.run([sys.executable, "-c", _VMAPPED, str(Path(__file__).resolve().parent.parent)], capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.split("\n")[:5] == [f"{c} raised True" for c in ("encode", "decode", "histogram", "pack", "unpack")]


@pytest.mark.gpu
def test_a_call_on_a_side_stream_does_not_wait_for_and_is_not_overwritten_by_the_current_one(dq):
    """The current stream is busy while the call runs on another: what the current stream has queued (here the fill of
    the guard words, done when an output is allocated) must not land on the results."""
    p = dq.DqParams(512, 2, 3)
    g = torch.randn(70_001, device="cuda")
    want = dq.dqsg_encode(g, 1, 0, 0, p)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    torch.cuda._sleep(20_000_000)                       # about ten milliseconds
    got = dq.dqsg_encode(g, 1, 0, 0, p, stream=side)
    with torch.cuda.stream(side):
        early = [t.cpu() for t in got]
    torch.cuda.synchronize()
    for w, e, t in zip(want, early, got):
        assert torch.equal(w.cpu(), e) and torch.equal(w, t)


@pytest.mark.gpu
def test_an_encode_without_a_gradient_leaves_the_buffers_alone(dq):
    p = dq.DqParams(512, 2, 3)
    pk, sc = torch.full((63,), 7, dtype=torch.int32, device="cuda"), torch.full((2,), 7.0, device="cuda")
    with pytest.raises(TypeError):
        dq.dqsg_encode(None, 1, 0, 0, p, pk, sc)
    assert bool((pk == 7).all()) and bool((sc == 7.0).all())
