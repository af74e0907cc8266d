"""The decoder's group sizes (8, 16 and 32 elements per lane, picked by length and worker count) at the lengths where
the choice changes, with ragged ends, odd bucket sizes and every code width: against the oracle on the ends and the
middle of the vector, bit for bit (every operation of the kernel rounds as the oracle's does)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from dq_testlib import gpu_encode, gpu_msg, oracle_msg, words_np  # noqa: E402
from dq_workloads.generators import DQSG, NDQSG, WorkerSpec  # noqa: E402
from test_gpu_parity import dq, oracle  # noqa: E402,F401


def _edges():
    sms = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 148
    wave8 = sms * 128 * 8 * 8                    # longest call of 8-element lanes
    two_and_a_half32 = sms * 128 * 32 * 5 * 5 // 2
    return {"8 last": wave8, "16 first": wave8 + 1, "16 last": two_and_a_half32 - 1, "32 first": two_and_a_half32 + 9,
            "16 last of all routines": 2 * wave8, "32 first of all routines": 2 * wave8 + 33,
            "8 last, many": wave8, "8 in seven CTAs, many": wave8 // 8 * 7}


@pytest.mark.parametrize("edge", ["8 last", "16 first", "16 last", "32 first", "16 last of all routines",
                                  "32 first of all routines", "8 last, many", "8 in seven CTAs, many"])
@pytest.mark.parametrize("bits,K,alpha,dither,bucket", [(1, 2, 1.0, 32, 96), (3, 8, 1.0, 16, 2048), (2, 3, 1.0, 32, 1024),
                                                        (2, 3, 1.0, 16, 992), (5, 21, 0.75, 32, 1248),
                                                        (7, 100, 1.0, 16, 32), (8, 128, 0.5, 32, 65536)])
def test_group_sizes_at_their_edges(dq, oracle, edge, bits, K, alpha, dither, bucket):
    n, step = _edges()[edge], 5
    rng = np.random.default_rng(bits)
    nested = 7 if "all routines" in edge else 9 if "many" in edge else 2
    specs = [WorkerSpec(DQSG, bits, 0, 0, 0.0, 1.0, 11, dither),
             *[WorkerSpec(NDQSG, bits, 0, K, float(K), alpha, 12 + w, dither) for w in range(nested)]]
    side = (0.01 * rng.standard_normal(n)).astype(np.float32)
    gmsgs, sent = [], []
    for w, sp in enumerate(specs):
        g = side + (0.0005 * rng.standard_normal(n)).astype(np.float32)
        pk, sc = gpu_encode(dq, torch, torch.from_numpy(g).cuda(), sp, w, step, bucket)
        gmsgs.append(gpu_msg(dq, pk, sc, sp, w, bucket))
        sent.append((words_np(pk), sc.cpu().numpy()))
    outs = {"vector": dq.ndqsg_decode_aggregate(gmsgs, n, step, torch.from_numpy(side).cuda())[:n].cpu().numpy(),
            "first": dq.ndqsg_decode_aggregate_side_first(gmsgs, n, step)[:n].cpu().numpy(),
            "running": dq.ndqsg_decode_aggregate_running(gmsgs, n, step)[:n].cpu().numpy()}
    # whole buckets at the start, in the middle and at the (ragged) end
    nb = -(-n // bucket)
    span = max(1, 4096 // bucket)
    for b0 in (0, nb // 2, max(0, nb - span)):
        lo, hi = b0 * bucket, min(n, (b0 + span) * bucket)
        omsgs = [oracle_msg(oracle, pk[lo * bits // 32:-(-hi * bits // 32)], sc[b0:b0 + span], sp, w, bucket)
                 for w, ((pk, sc), sp) in enumerate(zip(sent, specs))]
        y0 = oracle.decode_aggregate(omsgs[:1], hi - lo, step, i0=lo)
        want = {"vector": oracle.decode_aggregate(omsgs, hi - lo, step, side_info=side[lo:hi], i0=lo),
                "first": oracle.decode_aggregate(omsgs, hi - lo, step, side_info=y0, i0=lo),
                "running": oracle.decode_aggregate(omsgs, hi - lo, step, running=True, i0=lo)}
        for k, ref in want.items():
            assert np.array_equal(outs[k][lo:hi].view(np.uint32), ref.view(np.uint32)), (k, lo)


@pytest.mark.parametrize("workers,over", [(47, 33), (48, 0), (48, 33)])
@pytest.mark.parametrize("bits,dither", [(1, 32), (2, 16)])
def test_many_messages_take_long_groups_sooner(dq, oracle, workers, over, bits, dither):
    n, step, bucket = 4 * _edges()["16 last of all routines"] // 3 + over, 6, 992
    gen = torch.Generator(device="cuda").manual_seed(n)
    side = 0.01 * torch.randn(n, device="cuda", generator=gen)
    specs = [WorkerSpec(DQSG, bits, 0, 0, 0.0, 1.0, 11, dither),
             *[WorkerSpec(NDQSG, bits, 0, 1 << bits, float(1 << bits), 1.0, 12 + w, dither) for w in range(workers - 1)]]
    gmsgs, sent = [], []
    for w, sp in enumerate(specs):
        pk, sc = gpu_encode(dq, torch, side + 0.0005 * torch.randn(n, device="cuda", generator=gen), sp, w, step, bucket)
        gmsgs.append(gpu_msg(dq, pk, sc, sp, w, bucket))
        sent.append((pk, sc))
    outs = {"first": dq.ndqsg_decode_aggregate_side_first(gmsgs, n, step)[:n].cpu().numpy(),
            "running": dq.ndqsg_decode_aggregate_running(gmsgs, n, step)[:n].cpu().numpy()}
    nb = -(-n // bucket)
    for b0 in (0, nb - 3):
        lo, hi = b0 * bucket, min(n, (b0 + 3) * bucket)
        omsgs = [oracle_msg(oracle, words_np(pk[lo * bits // 32:-(-hi * bits // 32)]), sc[b0:b0 + 3].cpu().numpy(), sp, w, bucket)
                 for w, ((pk, sc), sp) in enumerate(zip(sent, specs))]
        y0 = oracle.decode_aggregate(omsgs[:1], hi - lo, step, i0=lo)
        want = {"first": oracle.decode_aggregate(omsgs, hi - lo, step, side_info=y0, i0=lo),
                "running": oracle.decode_aggregate(omsgs, hi - lo, step, running=True, i0=lo)}
        for k, ref in want.items():
            assert np.array_equal(outs[k][lo:hi].view(np.uint32), ref.view(np.uint32)), (k, lo)
