"""The forms in which the decoder joins code and dither (by kind, code width, dither stream and group size), bit for bit
against the oracle, at every group size, with scales from subnormal numbers to near the end of the fp32 range: beyond kappa_limit a
group is decoded by the plain routine."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from dq_testlib import gpu_encode, gpu_msg, oracle_msg, words_np  # noqa: E402
from dq_workloads.generators import DQSG, NDQSG, WorkerSpec  # noqa: E402
from test_gpu_parity import dq, oracle  # noqa: E402,F401

# factors of consecutive buckets: subnormal and tiny scales, ordinary ones, ones around the limits 2^114 to 2^120 and above
FACTORS = np.array([1.0, 1e-40, 1e-34, 0.0, 1.0, 1e30, 3e34, 2e35, 1e36, 4e36, 1.0, 1.5e37], np.float32)
BUCKET = 1248                                # (not a power of two, and buckets begin inside a warp's groups)


def _length(group):
    """A length that the decoder takes in groups of `group` elements per lane."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 148
    return {8: 12 * BUCKET + 77, 16: sms * 128 * 8 * 8 + 1, 32: sms * 128 * 32 * 5 * 5 // 2 + 1}[group]


@pytest.mark.parametrize("group,few", [(8, True), (8, False), (16, True), (16, False), (32, True)],
                         ids=["8", "8 many", "16", "16 many", "32"])
@pytest.mark.parametrize("dither,widths", [(32, (1, 2, 3, 4)), (16, (1, 2, 3, 4, 5, 6, 7, 8))])
def test_forms_over_the_range_of_scales(dq, oracle, group, few, dither, widths):
    n, step = _length(group), 9
    rng = np.random.default_rng(n + dither)
    nb = -(-n // BUCKET)
    common = rng.standard_normal(n).astype(np.float32)
    near = common + 0.05 * rng.standard_normal(n).astype(np.float32)
    for bits in widths if few else widths[1:3]:
        odd_K = (1 << bits) - 1 if bits > 1 else 2
        for K, M1, alpha in ((1 << bits, 2.0, 1.0), (odd_K, 0.01, 0.75), (odd_K, 2.0, 1.0), (1 << bits, 2.0, 0.75)):
            nested = 2 if few else 8
            # (no overflow in the sum: a step of the coarser quantizer is 75 scales)
            most = np.float32(2e35 if M1 < 1.0 else 1.5e37 if few else 4e36)
            factor = np.repeat(np.minimum(np.resize(FACTORS, nb), most), BUCKET)[:n]
            side = common * factor
            g_dev = torch.from_numpy(near * factor).cuda()
            specs = [WorkerSpec(DQSG, bits, 0, 0, 0.0, 1.0, 11, dither),
                     *[WorkerSpec(NDQSG, bits, 0, K, M1, alpha, 12 + w, dither) for w in range(nested)]]
            gmsgs, sent = [], []
            for w, sp in enumerate(specs):
                pk, sc = gpu_encode(dq, torch, g_dev, sp, w, step, BUCKET)
                gmsgs.append(gpu_msg(dq, pk, sc, sp, w, BUCKET))
                sent.append((words_np(pk), sc.cpu().numpy()))
            outs = {"one": dq.dqsg_decode_aggregate(gmsgs[:1], n, step)[:n].cpu().numpy(),
                    "dqsg": dq.dqsg_decode_aggregate([gmsgs[0]] * 2, n, step)[:n].cpu().numpy(),
                    "vector": dq.ndqsg_decode_aggregate(gmsgs, n, step, torch.from_numpy(side).cuda())[:n].cpu().numpy(),
                    "first": dq.ndqsg_decode_aggregate_side_first(gmsgs, n, step)[:n].cpu().numpy(),
                    "running": dq.ndqsg_decode_aggregate_running(gmsgs, n, step)[:n].cpu().numpy()}
            span = len(FACTORS)
            for b0 in sorted({0, max(0, nb - span)}):
                lo, hi = b0 * BUCKET, min(n, (b0 + span) * BUCKET)
                omsgs = [oracle_msg(oracle, pk[lo * bits // 32:-(-hi * bits // 32)], sc[b0:b0 + span], sp, w, BUCKET)
                         for w, ((pk, sc), sp) in enumerate(zip(sent, specs))]
                y0 = oracle.decode_aggregate(omsgs[:1], hi - lo, step, i0=lo)
                want = {"one": y0, "dqsg": oracle.decode_aggregate([omsgs[0]] * 2, hi - lo, step, i0=lo),
                        "vector": oracle.decode_aggregate(omsgs, hi - lo, step, side_info=side[lo:hi], i0=lo),
                        "first": oracle.decode_aggregate(omsgs, hi - lo, step, side_info=y0, i0=lo),
                        "running": oracle.decode_aggregate(omsgs, hi - lo, step, running=True, i0=lo)}
                for k, ref in want.items():
                    assert np.array_equal(outs[k][lo:hi].view(np.uint32), ref.view(np.uint32)), (k, bits, K, lo)


@pytest.mark.parametrize("exponent", [-119, -121, -125, -127, -140])
@pytest.mark.parametrize("dither,bits", [(32, 3), (32, 4), (16, 1), (16, 2), (16, 7)])
def test_a_fine_resolution_near_the_end_of_the_fp32_range(dq, oracle, dither, bits, exponent):
    """alpha M1 close to or among the subnormal numbers: scaled by less than one it would lose bits, and side information a
    few thousand steps long would be resolved to another coset."""
    n, step, M1 = 3 * BUCKET + 5, 4, float(np.ldexp(1.37, exponent))
    rng = np.random.default_rng(bits - exponent)
    grad = torch.from_numpy(np.float32(2.0 ** -98) * rng.standard_normal(n).astype(np.float32)).cuda()
    side = np.ldexp(rng.standard_normal(n), -96 - exponent + 12).astype(np.float32)
    for K, alpha in ((1 << bits, 1.0), (1 << bits, 0.75), ((1 << bits) - 1 if bits > 1 else 2, 1.0)):
        sp = WorkerSpec(NDQSG, bits, 0, K, M1, alpha, 21, dither)
        pk, sc = gpu_encode(dq, torch, grad, sp, 2, step, BUCKET)
        msg = gpu_msg(dq, pk, sc, sp, 2, BUCKET)
        got = dq.ndqsg_decode_aggregate([msg], n, step, torch.from_numpy(side).cuda())[:n].cpu().numpy()
        omsg = oracle_msg(oracle, words_np(pk), sc.cpu().numpy(), sp, 2, BUCKET)
        ref = oracle.decode_aggregate([omsg], n, step, side_info=side)
        assert np.isfinite(ref).all() and np.array_equal(got.view(np.uint32), ref.view(np.uint32)), (K, alpha)
