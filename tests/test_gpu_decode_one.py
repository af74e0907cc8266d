"""The decoder of one DQSG message: both dither streams and every code width with one and with four groups per lane, at the
lengths where that changes and with ragged ends, as a bucket range, and into an output that is 16- but not 32-byte aligned --
bit for bit against the oracle on the ends and the middle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from dq_testlib import oracle_encode, oracle_msg, spec_params, words_np  # noqa: E402
from dq_workloads.generators import DQSG, WorkerSpec  # noqa: E402
from test_gpu_parity import dq, oracle  # noqa: E402,F401


def _one_group_limit(dither):
    sms = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 148
    return sms * 1024 * (8 if dither == 16 else 10)


def _check(dq, oracle, n, bits, dither, bucket, first=0, shift=0):
    step, sp = 7, WorkerSpec(DQSG, bits, 0, 0, 0.0, 1.0, 41, dither)
    g = torch.randn(n, device="cuda", generator=torch.Generator(device="cuda").manual_seed(n + bits))
    p = spec_params(dq, sp, bucket)
    pk, sc = dq.dqsg_encode_range(g, first, sp.seed, 3, step, p)
    out = torch.full((n + 8,), 3.0, device="cuda")[shift:shift + n + 4]
    dq.ndqsg_decode_aggregate_range([dq.Message(pk, sc, sp.seed, 3, dq.DQ_KIND_DQSG, p)], n, first, step, None, out[:n])
    assert bool((out[n:] == 3.0).all())                       # nothing past the end
    got = out[:n].cpu().numpy()
    nb = -(-n // bucket)
    span = max(1, 8192 // bucket)
    for b0 in sorted({0, nb // 2, max(0, nb - span)}):        # whole buckets at the start, in the middle and at the end
        lo, hi = b0 * bucket, min(n, (b0 + span) * bucket)
        opk, osc = oracle_encode(oracle, g[lo:hi].cpu().numpy(), sp, 3, step, bucket, i0=first + lo)
        assert np.array_equal(words_np(pk)[lo * bits // 32:lo * bits // 32 + opk.size], opk)
        ref = oracle.decode_aggregate([oracle_msg(oracle, opk, osc, sp, 3, bucket)], hi - lo, step, i0=first + lo)
        assert np.array_equal(got[lo:hi].view(np.uint32), ref.view(np.uint32)), (lo, hi)


@pytest.mark.parametrize("bits", range(1, 9))
@pytest.mark.parametrize("dither", [32, 16])
def test_both_kernels_of_every_width(dq, oracle, dither, bits):
    limit = _one_group_limit(dither)
    for n, bucket in ((limit, 2048), (limit + 1, 96), (limit + 12_347, 1248), (70_007, 32), (5, 64), (1024 * 4 + 77, 65536)):
        _check(dq, oracle, n, bits, dither, bucket)


@pytest.mark.parametrize("bits,dither", [(1, 32), (3, 32), (5, 16), (8, 32), (7, 16)])
def test_a_bucket_range_and_an_output_between_32_byte_lines(dq, oracle, bits, dither):
    limit = _one_group_limit(dither)
    for n in (limit - 31, limit + 4099):
        _check(dq, oracle, n, bits, dither, 1248, first=1248 * 5_000_001, shift=4)
        _check(dq, oracle, n, bits, dither, 512, first=512 * 3, shift=4)
