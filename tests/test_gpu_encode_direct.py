"""The direct encoder where its shapes change: buckets within a chunk, a warp, a CTA and a cluster, bucket sizes that
leave idle lanes, the length at which a lane takes four groups instead of one, ragged ends, gradients that are 16- but
not 32-byte aligned, and the launch flags -- bit for bit against the oracle."""
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
