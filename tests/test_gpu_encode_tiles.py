"""The tile encoder, which takes long encodes that overlap by the launch flags in the lengths, power-of-two buckets and widths
of first_length: every mode, dither stream and code width, every bucket size, whole and ragged ends, bucket ranges and graph
capture.  The whole message against the unflagged call (the direct encoder's kernels), its ends and middle against the
oracle, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from dq_testlib import oracle_encode, words_np  # noqa: E402
from dq_workloads.generators import DQSG, NDQSG, WorkerSpec  # noqa: E402
from test_gpu_parity import dq, oracle  # noqa: E402,F401

BUCKETS = [32, 64, 128, 256, 512, 1024, 2048, 4096, 8192]


def first_length(bucket, bits):
    """The shortest gradient that the tile encoder takes, None where it takes none."""
    if bucket <= 256 or bits == 7:
        return 1 << 24
    if bucket == 8192:
        return 3 << 23 if bits in (5, 6) else None
    return {512: 1 << 25, 1024: 3 << 25, 2048: 1 << 26}.get(bucket)


WIDEST = 3 << 25


def _spec(mode, bits, dither):
    if mode == "dqsg":
        return WorkerSpec(DQSG, bits, 0, 0, 0.0, 1.0, 31, dither)
    K = {"pow2": 1 << bits, "mask": 1 << (bits - 1), "any": (1 << bits) - 1}[mode]
    return WorkerSpec(NDQSG, bits, 0, K, 1.5 * K, 0.9, 32, dither)


KERNELS = [(m, b, d) for m in ("dqsg", "pow2", "mask", "any") for b in range(1, 9) for d in (32, 16)
           if not (b == 1 and m in ("mask", "any"))]


@pytest.fixture(scope="module")
def gradient():
    gen = torch.Generator(device="cuda").manual_seed(77)
    return 0.01 * torch.randn(WIDEST + 10 * 8192, device="cuda", generator=gen)


def _takes_tiles(dq, g, spec, bucket):
    """Whether a flagged encode of `g` launches the tile encoder, the one with dynamic shared memory: from a captured graph."""
    from cuda.bindings import driver
    p = dq.binding.make_params(bucket, spec.bits, spec.levels, spec.coarse_K, spec.fine_M, spec.alpha, spec.dither_bits,
                               dq.DQ_FLAG_INPUT_READY | dq.DQ_FLAG_OUTPUT_FREE)
    out = dq.binding.alloc_message(g.numel(), p)
    encode = dq.dqsg_encode if spec.kind == DQSG else dq.ndqsg_encode
    encode(g, 1, 0, 0, p, *out)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        encode(g, 1, 0, 0, p, *out)
    raw = driver.CUgraph(graph.raw_cuda_graph())
    err, _, count = driver.cuGraphGetNodes(raw, 0)
    assert int(err) == 0 and count == 1
    err, nodes, _ = driver.cuGraphGetNodes(raw, 1)
    assert int(err) == 0
    err, params = driver.cuGraphKernelNodeGetParams(nodes[0])
    assert int(err) == 0
    return params.sharedMemBytes > 0


def _check(dq, oracle, g, spec, bucket, first=0, step=(1 << 33) + 6, worker=5):
    n, flags = g.numel(), dq.DQ_FLAG_INPUT_READY | dq.DQ_FLAG_OUTPUT_FREE
    encode = dq.dqsg_encode_range if spec.kind == DQSG else dq.ndqsg_encode_range
    got = []
    for f in (0, flags):
        p = dq.binding.make_params(bucket, spec.bits, spec.levels, spec.coarse_K, spec.fine_M, spec.alpha, spec.dither_bits, f)
        out = dq.binding.alloc_message(n, p)
        torch.cuda.synchronize()          # nothing before the flagged call touches its buffers
        got.append(encode(g, first, spec.seed, worker, step, p, *out))
    (pk, sc), (fpk, fsc) = got
    assert torch.equal(pk, fpk) and torch.equal(sc, fsc)
    span = 2 * max(bucket, 1024)          # (whole buckets)
    mid = n // 2 // span * span
    for lo, hi in ((0, span), (mid, mid + span), (n // span * span - span, n)):
        opk, osc = oracle_encode(oracle, g[lo:hi].cpu().numpy(), spec, worker, step, bucket, i0=first + lo)
        w0, b0 = lo * spec.bits // 32, lo // bucket
        assert np.array_equal(words_np(fpk[w0:w0 + opk.size]), opk), (lo, hi)
        assert np.array_equal(fsc[b0:b0 + osc.size].cpu().numpy().view(np.uint32), osc.view(np.uint32)), (lo, hi)


@pytest.mark.parametrize("k", range(len(KERNELS)))
def test_every_kernel(dq, oracle, gradient, k):
    mode, bits, dither = KERNELS[k]
    large = [b for b in BUCKETS[4:] if first_length(b, bits)]
    for bucket in (BUCKETS[k % 4], large[k % len(large)], 2048):       # within a warp's unit; in two halves
        _check(dq, oracle, gradient[:first_length(bucket, bits) + 12_345], _spec(mode, bits, dither), bucket)


@pytest.mark.parametrize("bucket", BUCKETS)
@pytest.mark.parametrize("more", [0, 1, 31, 33, 8192, 9 * 8192 + 8191])
def test_ends(dq, oracle, gradient, bucket, more):
    n = (1 << 24) + more
    for mode, bits, dither in (("dqsg", 3, 32), ("any", 2, 16)) if bucket <= 256 else (("dqsg", 7, 32), ("any", 7, 16)):
        _check(dq, oracle, gradient[:n], _spec(mode, bits, dither), bucket)


def test_a_bucket_range(dq, oracle, gradient):
    for bucket, bits in ((256, 3), (4096, 7)):
        _check(dq, oracle, gradient[:(1 << 24) + 77], _spec("pow2", bits, 32), bucket, first=bucket * 1_000_001)


@pytest.mark.parametrize("bucket", BUCKETS)
def test_the_shortest_gradients_of_the_tile_encoder_and_the_longest_of_the_other(dq, oracle, gradient, bucket):
    for bits in (2, 6, 7, 8):
        first, spec = first_length(bucket, bits), _spec("dqsg", bits, 32)
        for n in (WIDEST,) if first is None else (first - 1, first):
            assert _takes_tiles(dq, gradient[:n], spec, bucket) == (first is not None and n >= first), (bits, n)
            _check(dq, oracle, gradient[:n], spec, bucket)


@pytest.mark.parametrize("bucket,bits", [(256, 2), (2048, 7)])
def test_a_captured_sequence_replays_bit_identically(dq, gradient, bucket, bits):
    flags = dq.DQ_FLAG_INPUT_READY | dq.DQ_FLAG_OUTPUT_FREE
    n = first_length(bucket, bits) + 4321
    p = dq.binding.make_params(bucket, bits, 0, 1 << bits, 2.0, 1.0, 32, flags)
    grads = [gradient[:n], -gradient[:n], 0.5 * gradient[:n]]
    bufs = [dq.binding.alloc_message(n, p) for _ in grads]

    def encode():
        for w, (g, b) in enumerate(zip(grads, bufs)):
            dq.ndqsg_encode(g, 9, w, 3, p, *b)

    torch.cuda.synchronize()
    encode()
    torch.cuda.synchronize()
    want = [(pk.clone(), sc.clone()) for pk, sc in bufs]
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        encode()
    for _ in range(3):
        for pk, sc in bufs:
            pk.zero_()
            sc.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        for (pk, sc), (wpk, wsc) in zip(bufs, want):
            assert torch.equal(pk, wpk) and torch.equal(sc, wsc)
    assert dq.device_error_flags() == 0


@pytest.mark.parametrize("mode,bits,dither", [("mask", 8, 32), ("any", 8, 16), ("any", 8, 32), ("dqsg", 8, 32), ("mask", 7, 16),
                                              ("pow2", 8, 16), ("any", 5, 32), ("dqsg", 3, 16)])
@pytest.mark.parametrize("bucket", [128, 1024, 2048])
def test_many_launches_give_the_same_bits(dq, gradient, mode, bits, dither, bucket):
    _many_launches(dq, gradient, mode, bits, dither, bucket)


@pytest.mark.parametrize("mode,bits,dither", [("mask", 7, 16), ("any", 7, 32), ("dqsg", 7, 32), ("any", 5, 32), ("pow2", 6, 16)])
def test_many_launches_in_buckets_of_several_warps_give_the_same_bits(dq, gradient, mode, bits, dither):
    _many_launches(dq, gradient, mode, bits, dither, 8192)


def _many_launches(dq, gradient, mode, bits, dither, bucket):
    """A row must be in registers before its stage takes the next copy: where it was not, one launch in a few hundred had
    codes of the wrong elements at the ends of some rows."""
    n = first_length(bucket, bits)
    sp, g = _spec(mode, bits, dither), gradient[:n]
    encode = dq.dqsg_encode if sp.kind == DQSG else dq.ndqsg_encode
    make = lambda f: dq.binding.make_params(bucket, bits, sp.levels, sp.coarse_K, sp.fine_M, sp.alpha, dither, f)  # noqa: E731
    want = encode(g, 3, 1, 2, make(0))
    p = make(dq.DQ_FLAG_INPUT_READY | dq.DQ_FLAG_OUTPUT_FREE)
    out = dq.binding.alloc_message(n, p)
    wrong = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(1000):
        encode(g, 3, 1, 2, p, *out)
        wrong += (out[0] != want[0]).sum() + (out[1] != want[1]).sum()
    assert int(wrong) == 0
