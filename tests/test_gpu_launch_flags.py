"""Encodes that overlap by the launch flags, on message buffers that are used again and again with other contents: the
flags speak about the previous kernel only, so a kernel that stores without waiting must not run beside one that is two
launches back."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from test_gpu_parity import dq  # noqa: E402,F401

# around one CTA per SM, one and several waves, a cluster per bucket, long gradients, and the tile encoder
SHAPES = [(65_536, 512), (70_001, 32), (266_610, 1024), (300_000, 65536), (1_100_000, 2048), (1_663_370, 16384),
          (4_194_304, 4096), (17_000_000, 2048), (17_000_000, 256)]
ROUNDS = 6


def _params(dq, w, bucket, flags):
    q = (3, 5, 0, 0.0) if w == 0 else (2, 0, 4, 2.0)
    return dq.binding.make_params(bucket, *q, 0.0, 32, flags)


def _encode(dq, w, bucket, flags, grad, step, buf):
    fn = dq.dqsg_encode if w == 0 else dq.ndqsg_encode
    fn(grad, 50 + w, w, step, _params(dq, w, bucket, flags), *buf)


@pytest.mark.parametrize("n,bucket", SHAPES)
def test_flagged_steps_on_reused_buffers_give_the_means_of_plain_steps(dq, n, bucket):
    ready, free = dq.DQ_FLAG_INPUT_READY, dq.DQ_FLAG_OUTPUT_FREE
    W = 3
    gen = torch.Generator(device="cuda").manual_seed(n)
    common = torch.randn(n, device="cuda", generator=gen)
    grads = [[common + 0.1 * torch.randn(n, device="cuda", generator=gen) for _ in range(W)] for _ in range(ROUNDS)]
    bufs = [dq.binding.alloc_message(n, _params(dq, w, bucket, 0)) for w in range(W)]
    msgs = [dq.Message(*bufs[w], 50 + w, w, int(w > 0), _params(dq, w, bucket, 0)) for w in range(W)]
    means = {k: [torch.empty(n, device="cuda") for _ in range(ROUNDS)] for k in ("plain", "flagged")}
    torch.cuda.synchronize()
    for kind in ("plain", "flagged", "flagged"):
        for i in range(ROUNDS):
            for w in range(W):
                flags = 0 if kind == "plain" else ready | (free if w > 0 else 0)
                _encode(dq, w, bucket, flags, grads[i][w], i, bufs[w])
            dq.ndqsg_decode_aggregate_side_first(msgs, n, i, means[kind][i])
        torch.cuda.synchronize()
        if kind == "flagged":
            for i in range(ROUNDS):
                assert torch.equal(means["plain"][i], means["flagged"][i]), i
                means["flagged"][i].zero_()
            torch.cuda.synchronize()
    assert dq.device_error_flags() == 0


@pytest.mark.parametrize("n,bucket", SHAPES)
def test_two_buffers_used_in_turn_hold_the_last_messages(dq, n, bucket):
    both = dq.DQ_FLAG_INPUT_READY | dq.DQ_FLAG_OUTPUT_FREE
    grads = [torch.randn(n, device="cuda") for _ in range(4)]
    want = [dq.ndqsg_encode(g, 51, 1, i, _params(dq, 1, bucket, 0)) for i, g in enumerate(grads)]
    bufs = [dq.binding.alloc_message(n, _params(dq, 1, bucket, 0)) for _ in range(2)]
    torch.cuda.synchronize()
    for rep in range(4):
        for i in range(4):
            _encode(dq, 1, bucket, both, grads[i], i, bufs[i % 2])
        torch.cuda.synchronize()
        for i in (2, 3):
            assert torch.equal(bufs[i % 2][0], want[i][0]) and torch.equal(bufs[i % 2][1], want[i][1]), (rep, i)
