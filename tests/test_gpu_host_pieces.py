"""The host-buffer calls: without copies (short, pinned, aligned), in pieces on two streams (long), and with plain copies
(pageable or misaligned buffers) give the bits of the device calls."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from test_gpu_parity import dq  # noqa: E402,F401

DIRECT, PIECES = 1 << 20, 1 << 22


def _host(t, how):
    """`t` as a host tensor: pinned, pageable, or pinned 4 bytes past an aligned address."""
    n = t.numel()
    if how == "pageable":
        h = torch.empty(n, dtype=t.dtype)
    elif how == "pinned":
        h = torch.empty(n, dtype=t.dtype).pin_memory()
    else:
        h = torch.empty(n + 1, dtype=t.dtype).pin_memory()[1:]
    return h.copy_(t)


@pytest.mark.parametrize("how", ["pinned", "pageable", "misaligned"])
@pytest.mark.parametrize("n,bucket", [(1, 32), (70_001, 512), (DIRECT, 2048), (DIRECT + 1, 2048), (PIECES - 1, 4096),
                                      (PIECES, 65536), (PIECES + 777, 96), (5_000_011, 8192)])
def test_host_calls_give_the_bits_of_the_device_calls(dq, n, bucket, how):
    torch.manual_seed(n + bucket)
    first, rest = dq.DqParams(bucket, 3, 5, 0, 0, 0, 32, 0), dq.DqParams(bucket, 2, 0, 3, 3.0, 0, 32, 0)
    common = 0.01 * torch.randn(n, device="cuda")
    dev, host, ws = [], [], torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
    for w in range(3):
        p, nd = (first, False) if w == 0 else (rest, True)
        g = common + 0.001 * torch.randn(n, device="cuda")
        pk, sc = dq.binding.alloc_message(n, p)
        (dq.ndqsg_encode if nd else dq.dqsg_encode)(g, 40 + w, w, 2, p, pk, sc)
        hpk, hsc = _host(torch.zeros_like(pk), how), _host(torch.zeros_like(sc), how)
        (dq.ndqsg_encode_host if nd else dq.dqsg_encode_host)(_host(g, how), 40 + w, w, 2, p, hpk, hsc, ws)
        assert torch.equal(hpk, pk.cpu()) and torch.equal(hsc, sc.cpu())
        dev.append(dq.Message(pk, sc, 40 + w, w, int(nd), p))
        host.append(dq.Message(hpk, hsc, 40 + w, w, int(nd), p))
    out = _host(torch.zeros(n), how)
    dq.ndqsg_decode_aggregate_side_first_host(host, n, 2, out, ws)
    assert torch.equal(out, dq.ndqsg_decode_aggregate_side_first(dev, n, 2)[:n].cpu())
    out.zero_()
    dq.ndqsg_decode_aggregate_host(host, n, 2, _host(common, how), out, ws)
    assert torch.equal(out, dq.ndqsg_decode_aggregate(dev, n, 2, common)[:n].cpu())
