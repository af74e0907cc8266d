"""The tile encoder, which takes encodes of 2^24 elements and more that overlap by the launch flags (power-of-two buckets
up to 8192): every mode, dither stream and code width, every bucket size, whole and ragged ends, bucket ranges and graph
capture.  The whole message against the unflagged call (the direct encoder's kernels), its ends and middle against the
oracle, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from dq_testlib import oracle_encode, words_np  # noqa: E402
from dq_workloads.generators import DQSG, NDQSG, WorkerSpec  # noqa: E402
from test_gpu_parity import dq, oracle  # noqa: E402,F401

FIRST = 1 << 24                           # shortest gradient that the tile encoder takes
BUCKETS = [32, 64, 128, 256, 512, 1024, 2048, 4096, 8192]


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
    return 0.01 * torch.randn(FIRST + 10 * 8192, device="cuda", generator=gen)


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
    for bucket in (BUCKETS[k % 6], BUCKETS[6 + k % 3]):                # one within a warp's unit, one in two halves
        _check(dq, oracle, gradient[:FIRST + 12_345], _spec(mode, bits, dither), bucket)


@pytest.mark.parametrize("bucket", BUCKETS)
@pytest.mark.parametrize("more", [0, 1, 31, 33, 8192, 9 * 8192 + 8191])
def test_ends(dq, oracle, gradient, bucket, more):
    _check(dq, oracle, gradient[:FIRST + more], _spec("dqsg", 3, 32), bucket)
    _check(dq, oracle, gradient[:FIRST + more], _spec("any", 2, 16), bucket)


def test_a_bucket_range(dq, oracle, gradient):
    for bucket in (512, 4096):
        _check(dq, oracle, gradient[:FIRST + 77], _spec("pow2", 3, 32), bucket, first=bucket * 1_000_001)


def test_the_shortest_gradient_of_the_tile_encoder_and_the_longest_of_the_other(dq, oracle, gradient):
    for n in (FIRST - 1, FIRST):
        _check(dq, oracle, gradient[:n], _spec("dqsg", 2, 32), 2048)


def test_a_captured_sequence_replays_bit_identically(dq, gradient):
    flags = dq.DQ_FLAG_INPUT_READY | dq.DQ_FLAG_OUTPUT_FREE
    n = FIRST + 4321
    p = dq.binding.make_params(2048, 2, 0, 4, 2.0, 1.0, 32, flags)
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
@pytest.mark.parametrize("bucket", [1024, 2048, 8192])
def test_many_launches_give_the_same_bits(dq, gradient, mode, bits, dither, bucket):
    """A row must be in registers before its stage takes the next copy: where it was not, one launch in a few hundred had
    codes of the wrong elements at the ends of some rows."""
    sp, g = _spec(mode, bits, dither), gradient[:FIRST]
    encode = dq.dqsg_encode if sp.kind == DQSG else dq.ndqsg_encode
    make = lambda f: dq.binding.make_params(bucket, bits, sp.levels, sp.coarse_K, sp.fine_M, sp.alpha, dither, f)  # noqa: E731
    want = encode(g, 3, 1, 2, make(0))
    p = make(dq.DQ_FLAG_INPUT_READY | dq.DQ_FLAG_OUTPUT_FREE)
    out = dq.binding.alloc_message(FIRST, p)
    wrong = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(1000):
        encode(g, 3, 1, 2, p, *out)
        wrong += (out[0] != want[0]).sum() + (out[1] != want[1]).sum()
    assert int(wrong) == 0
