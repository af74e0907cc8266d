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


@pytest.mark.parametrize("how,in_place", [("pinned", True), ("end of a block", True), ("registered", True), ("pageable", False),
                                          ("misaligned", False)])
def test_the_workspace_stays_untouched_where_the_buffers_are_used_in_place(dq, how, in_place):
    """... and nowhere else.  `registered`: page-locked by registration of exactly the buffer's pages."""
    n, p = 8192, dq.DqParams(512, 2, 3, 0, 0, 0, 32, 0)
    g = torch.randn(n, device="cuda")
    want = dq.dqsg_encode(g, 3, 0, 1, p)
    registered = []

    def host(t):
        if how == "end of a block":                       # nothing behind the buffer in its page-locked block
            h = torch.empty((1 << 20) // t.element_size(), dtype=t.dtype).pin_memory()[-t.numel():]
        elif how == "registered":
            page = torch.empty(4096 * 17, dtype=torch.uint8)
            at = -page.data_ptr() % 4096
            size = -(-t.numel() * t.element_size() // 4096) * 4096
            h = page[at:at + size].view(t.dtype)[-t.numel():]
            assert int(torch.cuda.cudart().cudaHostRegister(page.data_ptr() + at, size, 0)) == 0
            registered.append((page.data_ptr() + at, page))       # (the pages live until they are unregistered)
        else:
            h = _host(t, how)
        return h.copy_(t)

    ws = torch.full((1 << 20,), 0x5A, dtype=torch.uint8, device="cuda")
    pk, sc = host(torch.zeros(n // 16, dtype=torch.int32)), host(torch.zeros(16))
    try:
        dq.dqsg_encode_host(host(g.cpu()), 3, 0, 1, p, pk, sc, ws)
        assert torch.equal(pk, want[0].cpu()) and torch.equal(sc, want[1].cpu())
        assert bool((ws == 0x5A).all()) == in_place
        out = host(torch.zeros(n))
        ws.fill_(0x5A)
        dq.ndqsg_decode_aggregate_host([dq.Message(pk, sc, 3, 0, 0, p)], n, 1, None, out, ws)
        assert torch.equal(out, dq.dqsg_decode_aggregate([dq.Message(*want, 3, 0, 0, p)], n, 1)[:n].cpu())
        assert bool((ws == 0x5A).all()) == in_place
    finally:
        for address, _ in registered:
            torch.cuda.cudart().cudaHostUnregister(address)


@pytest.mark.parametrize("n,bits", [(70_001, 2), (70_001, 3), (5_000_011, 2), (18_000_000, 2)])
def test_the_launch_flags_mean_nothing_to_host_calls(dq, n, bits):
    """A short call in place directly follows the caller's previous kernel, which may still use the workspace: here it
    copies from it, and must find what was there."""
    flags = dq.DQ_FLAG_INPUT_READY | dq.DQ_FLAG_OUTPUT_FREE
    p, pf = dq.DqParams(2048, bits, 3, 0, 0, 0, 32, 0), dq.DqParams(2048, bits, 3, 0, 0, 0, 32, flags)
    g = torch.randn(n, device="cuda")
    pk, sc = dq.dqsg_encode(g, 3, 0, 1, p)
    host = _host(g, "pinned"), _host(torch.zeros_like(pk), "pinned"), _host(torch.zeros_like(sc), "pinned")
    ws = torch.empty(dq.encode_workspace_bytes(n, p), dtype=torch.uint8, device="cuda")
    for _ in range(3):
        ws.fill_(0x5A)
        hist = dq.code_histogram(ws.view(torch.int32), ws.numel() // 4, 8)
        dq.dqsg_encode_host(host[0], 3, 0, 1, pf, host[1], host[2], ws)
        assert torch.equal(host[1], pk.cpu()) and torch.equal(host[2], sc.cpu())
        assert int(hist[0x5A]) == ws.numel() // 4


@pytest.mark.parametrize("bits", range(1, 9))
def test_codes_that_would_cross_the_bus_in_small_pieces_go_through_the_workspace(dq, bits):
    n, p = 70_001, dq.DqParams(512, bits, 0, 0, 0, 0, 32, 0)
    g = torch.randn(n, device="cuda")
    pk, sc = dq.dqsg_encode(g, 3, 0, 1, p)
    ws = torch.full((1 << 20,), 0x5A, dtype=torch.uint8, device="cuda")
    hpk, hsc = _host(torch.zeros_like(pk), "pinned"), _host(torch.zeros_like(sc), "pinned")
    dq.dqsg_encode_host(_host(g, "pinned"), 3, 0, 1, p, hpk, hsc, ws)
    assert torch.equal(hpk, pk.cpu()) and torch.equal(hsc, sc.cpu())
    used = ws.cpu() != 0x5A
    assert bool(used.any()) == (bits in (3, 5, 6, 7))
    assert not bool(used[4 * pk.numel():].any())
