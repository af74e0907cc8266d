"""The direct encoder where its shapes change: buckets within a chunk, a warp, a CTA and a cluster, bucket sizes that
leave idle lanes, the length at which a lane takes four groups instead of one, the grids that take the kernels with fewer
registers, ragged ends, gradients that are 16- but not 32-byte aligned, and the launch flags -- bit for bit against the
oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from dq_testlib import gpu_encode, oracle_encode, words_np  # noqa: E402
from dq_workloads.generators import DQSG, NDQSG, WorkerSpec  # noqa: E402
from test_gpu_parity import dq, oracle  # noqa: E402,F401

SPECS = [WorkerSpec(DQSG, 1, 2, 0, 0.0, 1.0, 21, 32), WorkerSpec(DQSG, 3, 5, 0, 0.0, 1.0, 22, 16),
         WorkerSpec(NDQSG, 2, 0, 3, 3.0, 1.0, 23, 32), WorkerSpec(NDQSG, 7, 0, 100, 64.0, 0.75, 24, 16),
         WorkerSpec(NDQSG, 8, 0, 32, 16.0, 1.0, 25, 32)]


def _one_group_limit():
    return torch.cuda.get_device_properties(0).multi_processor_count * 1024 * 8 if torch.cuda.is_available() else 1212416


def _check(dq, oracle, g, gd, sp, bucket, step=3):
    pk, sc = gpu_encode(dq, torch, gd, sp, 4, step, bucket)
    opk, osc = oracle_encode(oracle, g, sp, 4, step, bucket, threads=8)
    assert np.array_equal(words_np(pk), opk)
    assert np.array_equal(sc.cpu().numpy().view(np.uint32), osc.view(np.uint32))


@pytest.mark.parametrize("bucket", [32, 96, 224, 256, 288, 512, 1024, 1056, 2048, 2080, 4096, 4128, 8192, 8224, 12288, 16416,
                                    32768, 65504, 65536])
@pytest.mark.parametrize("over", [-1, 1])           # last length with one group per lane; one past it, with four
def test_bucket_shapes(dq, oracle, bucket, over):
    n = _one_group_limit() if over < 0 else _one_group_limit() + 8 * 37 + 5
    g = (0.01 * np.random.default_rng(bucket).standard_normal(n)).astype(np.float32)
    sp = SPECS[(bucket // 32 + over) % len(SPECS)]
    _check(dq, oracle, g, torch.from_numpy(g).cuda(), sp, bucket)


@pytest.mark.parametrize("spec", range(len(SPECS)))
@pytest.mark.parametrize("n", [1, 7, 8, 9, 31, 33, 1023, 65536 + 40, 1_400_003])
def test_lengths_and_alignment(dq, oracle, spec, n):
    g = (0.01 * np.random.default_rng(n).standard_normal(n)).astype(np.float32)
    shifted = torch.empty(n + 4, dtype=torch.float32, device="cuda")[4:]       # 16 bytes past an aligned address
    shifted.copy_(torch.from_numpy(g))
    for bucket in (160, 2048):
        _check(dq, oracle, g, shifted, SPECS[spec], bucket)


@pytest.mark.parametrize("n,bucket", [(70_001, 512), (3_000_000, 2048), (3_000_001, 65536), (17_000_000, 4096)])
def test_overlapping_launches_give_the_bits_of_plain_ones(dq, oracle, n, bucket):
    p = dq.binding.make_params(bucket, 2, 3)
    both = dq.binding.make_params(bucket, 2, 3, flags=dq.DQ_FLAG_INPUT_READY | dq.DQ_FLAG_OUTPUT_FREE)
    grads = [0.01 * torch.randn(n, device="cuda") for _ in range(3)]
    plain = [dq.dqsg_encode(g, 9, w, 1, p) for w, g in enumerate(grads)]
    torch.cuda.synchronize()
    over = [dq.binding.alloc_message(n, both) for _ in grads]
    torch.cuda.synchronize()
    for _ in range(3):
        for w, g in enumerate(grads):
            dq.dqsg_encode(g, 9, w, 1, both, *over[w])
    avg = dq.dqsg_decode_aggregate([dq.Message(pk, sc, 9, w, dq.DQ_KIND_DQSG, p) for w, (pk, sc) in enumerate(over)], n, 1)
    ref = dq.dqsg_decode_aggregate([dq.Message(pk, sc, 9, w, dq.DQ_KIND_DQSG, p) for w, (pk, sc) in enumerate(plain)], n, 1)
    assert torch.equal(avg, ref)
    for (pk, sc), (pk0, sc0) in zip(over, plain):
        assert torch.equal(pk, pk0) and torch.equal(sc, sc0)


KERNELS = [(m, b, d) for m in ("dqsg", "pow2", "mask", "any") for b in range(1, 9) for d in (32, 16)
           if not (b == 1 and m in ("mask", "any"))]


@pytest.mark.parametrize("k", range(len(KERNELS)))
def test_grids_that_take_the_dense_kernels(dq, oracle, k):
    """One wave of CTAs with 64 (one group per lane: 40) registers that would be two with 80 (48), buckets in clusters, and
    more waves of windows whose buckets share warps."""
    mode, bits, dither = KERNELS[k]
    sms = _one_group_limit() // 8192
    K = {"dqsg": 0, "pow2": 1 << bits, "mask": 1 << (bits - 1), "any": (1 << bits) - 1}[mode]
    sp = WorkerSpec(NDQSG if K else DQSG, bits, 0, K, 1.5 * K, 0.9 if K else 1.0, 33, dither)
    flags = dq.DQ_FLAG_INPUT_READY | dq.DQ_FLAG_OUTPUT_FREE if k % 2 else 0
    encode = dq.ndqsg_encode if K else dq.dqsg_encode
    for n, bucket in ((6 * sms * 4096 + 4099, 2048), (8192 * sms - 77, 12288), (sms * 10 * 2080 * 4 + 1, 2080),
                      (51 * 65536 + 31, 65536)):
        g = 0.01 * torch.randn(n, device="cuda", generator=torch.Generator(device="cuda").manual_seed(n))
        p = dq.binding.make_params(bucket, bits, sp.levels, sp.coarse_K, sp.fine_M, sp.alpha, dither, flags)
        out = dq.binding.alloc_message(n, p)
        torch.cuda.synchronize()
        pk, sc = encode(g, sp.seed, 4, 3, p, *out)
        nb = -(-n // bucket)
        span = max(1, 8192 // bucket)
        for b0 in sorted({0, nb // 2, nb - span}):
            lo, hi = b0 * bucket, min(n, (b0 + span) * bucket)
            opk, osc = oracle_encode(oracle, g[lo:hi].cpu().numpy(), sp, 4, 3, bucket, i0=lo, threads=8)
            assert np.array_equal(words_np(pk)[lo * bits // 32:lo * bits // 32 + opk.size], opk), (n, lo)
            assert np.array_equal(sc[b0:b0 + osc.size].cpu().numpy().view(np.uint32), osc.view(np.uint32)), (n, lo)
