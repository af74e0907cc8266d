"""The work that users of this library have it do, as cases that can be timed: per-worker encodes, the server's
decode-and-average, whole steps of both, the host-buffer calls, and the rate accounting and radix-3 container of a
finished message.

The sizes are those of the repository's own workloads and of the networks whose gradients the paper counts
(266,610 to 124,439,808 elements, and the sweep's 2^16 to 2^27 between and around them).  Gradients are normal,
Laplace or layered (one standard deviation per layer), the workers of a case are correlated as data-parallel
workers are.  Everything is drawn on the GPU from the seed.
"""
import math

import torch

import paper_1904_01197_b200 as dq

# Quantizer settings by name: kind, bits, levels (DQSG), coarse ratio K and fine resolution M1 (NDQSG).
QUANT = {
    "dqsg1": dict(kind=dq.DQ_KIND_DQSG, bits=1, levels=2),            # sign-like, two levels
    "dqsg2": dict(kind=dq.DQ_KIND_DQSG, bits=2, levels=3),            # the paper's three-level quantizer
    "dqsg3": dict(kind=dq.DQ_KIND_DQSG, bits=3, levels=5),            # the paper's five-level quantizer (M = 2)
    "dqsg4": dict(kind=dq.DQ_KIND_DQSG, bits=4, levels=15),
    "dqsg8": dict(kind=dq.DQ_KIND_DQSG, bits=8, levels=255),
    "ndqsg1": dict(kind=dq.DQ_KIND_NDQSG, bits=1, K=2, M=2.0),
    "ndqsg2": dict(kind=dq.DQ_KIND_NDQSG, bits=2, K=4, M=2.0),        # two bits sent instead of three
    "ndqsg2_k3": dict(kind=dq.DQ_KIND_NDQSG, bits=2, K=3, M=3.0),     # the paper's steps 1/3 and 1
    "ndqsg3": dict(kind=dq.DQ_KIND_NDQSG, bits=3, K=8, M=16.0),
    "ndqsg4": dict(kind=dq.DQ_KIND_NDQSG, bits=4, K=16, M=16.0),
}
STEP = 1       # training iteration: part of every dither counter


def listed():
    return [
        # The smallest call sequence: two workers' encodes and their fused decode on a gradient of 65,536 elements.
        # Launches and host work decide here, as they do for a small model or one layer at a time.
        dict(name="step_tiny", op="step", n=65536, workers=2, bucket=512, quant="ndqsg2", first="dqsg2",
             side="vector", dither=32, values="normal", overlap=False),
        # One worker's message for the paper's 300-100 fully connected network: small, with a ragged end.
        dict(name="encode_fc300", op="encode", n=266610, bucket=1024, quant="dqsg2", dither=32, values="normal"),
        # The paper's own nested setting (K = 3, not a power of two) on its LeNet-like network, a few large
        # partitions with one scale each.
        dict(name="encode_lenet_k3", op="encode", n=1663370, bucket=16384, quant="ndqsg2_k3", dither=32,
             values="normal"),
        # An ordinary encode: ResNet-18-sized, one standard deviation per layer.
        dict(name="encode_resnet18", op="encode", n=11689512, bucket=2048, quant="dqsg2", dither=32,
             values="layered"),
        # The largest encode: GPT-2-small-sized, three bits sent.
        dict(name="encode_gpt2", op="encode", n=124439808, bucket=4096, quant="ndqsg3", dither=32, values="laplace"),
        # Algorithm 2 as the paper writes it, on a small network: eight workers, the first half DQSG, the second
        # half NDQSG against the running mean.
        dict(name="decode_fc300_running", op="decode", n=266610, workers=8, firsts=4, bucket=1024,
             quant="ndqsg2_k3", first="dqsg3", side="running", dither=32, values="normal"),
        # A server that decodes one worker's message alone, e.g. to have the side information as a vector.
        dict(name="decode_resnet50_w1", op="decode", n=25557032, workers=1, firsts=1, bucket=2048, quant="dqsg3",
             first="dqsg3", side="none", dither=32, values="normal"),
        # The mean of eight DQSG messages (Algorithm 1) with the cheaper 16-bit dither stream.
        dict(name="decode_resnet18_d16", op="decode", n=11689512, workers=8, firsts=8, bucket=2048, quant="dqsg2",
             first="dqsg2", side="none", dither=16, values="layered"),
        # The largest decode: sixteen nested messages against a side-information vector.
        dict(name="decode_gpt2_w16", op="decode", n=124439808, workers=16, firsts=0, bucket=4096, quant="ndqsg3",
             first="dqsg3", side="vector", dither=32, values="laplace"),
        # A whole training step's communication, ResNet-50-sized: eight encodes back to back (with the launch flags
        # that back-to-back encodes of different gradients allow) and the fused decode that takes its side
        # information from worker 0.
        dict(name="step_resnet50", op="step", n=25557032, workers=8, bucket=2048, quant="ndqsg2", first="dqsg3",
             side="first", dither=32, values="normal", overlap=True),
        # The same path for a caller whose gradients and messages live in pinned host memory: one worker's encode,
        # then the server's decode of four messages.
        dict(name="host_resnet18", op="host", n=11689512, workers=4, bucket=2048, quant="ndqsg2", first="dqsg3",
             dither=32, values="normal"),
        # Rate accounting and the 1.6-bit container of a finished three-level message.
        dict(name="wire_resnet18", op="wire", n=11689512, bucket=2048, quant="dqsg2", dither=32, values="normal"),
    ]


def draw(rng):
    def log_int(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        if rng.random() < 0.25:
            n = (n + 4095) // 4096 * 4096          # a padded, even length
        return min(hi, max(lo, n))

    op = rng.choices(["encode", "decode", "step", "host", "wire"], weights=[8, 8, 4, 1, 2])[0]
    dither = rng.choices([32, 16], weights=[3, 1])[0]
    values = rng.choice(["normal", "laplace", "layered"])
    if rng.random() < 0.75:
        bucket = rng.choice([256, 512, 1024, 2048, 4096, 8192])
    else:
        bucket = 32 * int(round(math.exp(rng.uniform(0.0, math.log(2048)))))     # any multiple of 32 up to 65536
    dqsg = ["dqsg1", "dqsg2", "dqsg3", "dqsg4", "dqsg8"]
    nested = ["ndqsg1", "ndqsg2", "ndqsg2_k3", "ndqsg3", "ndqsg4"]
    case = dict(op=op, bucket=bucket, dither=dither, values=values)
    if op == "encode":
        case.update(n=log_int(1 << 16, 1 << 27), quant=rng.choice(dqsg + nested))
    elif op == "wire":
        case.update(n=log_int(1 << 16, 1 << 25), quant=rng.choices(["dqsg2", "dqsg1", "dqsg3", "ndqsg4"],
                                                                   weights=[4, 1, 1, 1])[0])
    elif op == "decode":
        workers = rng.choice([1, 2, 3, 4, 6, 8, 12, 16, 32])
        side = rng.choice(["none", "vector", "first", "running"]) if workers > 1 else "none"
        firsts = {"none": workers, "vector": rng.choice([0, workers // 2]), "first": 1,
                  "running": max(1, workers // 2)}[side]
        case.update(n=log_int(1 << 16, (1 << 29) // workers if workers > 8 else 1 << 26), workers=workers,
                    firsts=firsts, quant=rng.choice(nested), first=rng.choice(dqsg), side=side)
    else:
        case.update(n=log_int(1 << 16, 1 << 23), workers=rng.choice([2, 3, 4, 8]), quant=rng.choice(nested),
                    first=rng.choice(dqsg))
        if op == "step":
            case.update(side=rng.choice(["vector", "first", "running"]), overlap=False)
    return case


# ------------------------------------------------------------------------------------------------------ inputs
def _params(case, quant, flags=0):
    q = QUANT[quant]
    return dq.DqParams(case["bucket"], q["bits"], q.get("levels", 0), q.get("K", 0), q.get("M", 0.0), 0.0,
                       case["dither"], flags)


def _workers(case):
    """[(quantizer name, kind, dither seed)] in array order: the DQSG workers come first."""
    op = case["op"]
    if op in ("encode", "wire"):
        names = [case["quant"]]
    else:
        firsts = case["firsts"] if op == "decode" else 1
        names = [case["first"]] * firsts + [case["quant"]] * (case["workers"] - firsts)
    return [(q, QUANT[q]["kind"], 0x9E3779B97F4A7C15 * (w + 1) & 0xFFFFFFFFFFFFFFFF) for w, q in enumerate(names)]


class _Gradients:
    """The workers' gradients: a common part and a tenth of its variance of each worker's own."""

    def __init__(self, case, seed):
        self.n, self.values = case["n"], case["values"]
        self.gen = torch.Generator(device="cuda").manual_seed(seed)
        self.sigma = None
        if self.values == "layered":
            cuts = torch.rand(62, device="cuda", generator=self.gen).mul_(self.n).long().sort().values
            layer = torch.bucketize(torch.arange(self.n, device="cuda"), cuts, out_int32=True)
            sig = torch.exp(torch.empty(63, device="cuda").uniform_(math.log(1e-4), math.log(1e-1),
                                                                    generator=self.gen))
            self.sigma = sig[layer]
        self.common = self._unit(self.values)

    def _unit(self, values):
        if values == "laplace":
            x = torch.empty(self.n, device="cuda").exponential_(generator=self.gen)
            x -= torch.empty(self.n, device="cuda").exponential_(generator=self.gen)
            return x
        return torch.randn(self.n, device="cuda", generator=self.gen)

    def _scaled(self, x):
        return x.mul_(self.sigma) if self.sigma is not None else x.mul_(1e-2)

    def worker(self):
        x = torch.randn(self.n, device="cuda", generator=self.gen)
        return self._scaled(x.mul_(1.0 / 3.0).add_(self.common))

    def side(self):
        x = torch.randn(self.n, device="cuda", generator=self.gen)
        return self._scaled(x.mul_(0.05).add_(self.common))


def _message_buffers(n, params, pinned=False):
    where = dict(pin_memory=True) if pinned else dict(device="cuda")
    return (torch.empty(dq.packed_words(n, params.bits), dtype=torch.int32, **where),
            torch.empty(dq.num_buckets(n, params.bucket), dtype=torch.float32, **where))


def _encoder(kind):
    return dq.ndqsg_encode if kind == dq.DQ_KIND_NDQSG else dq.dqsg_encode


def prepare(case, seed):
    op, n = case["op"], case["n"]
    g = _Gradients(case, seed)
    s = {"case": case, "op": op, "n": n}
    workers = _workers(case)
    if op in ("encode", "step"):
        s["grads"], s["params"], s["msgs"] = [], [], []
        for w, (q, kind, dseed) in enumerate(workers):
            # the gradients of a step were complete before the first encode; the later encodes of an overlapping
            # step also write message buffers that the encode before them does not touch
            flags = 0
            if case.get("overlap"):
                flags = dq.DQ_FLAG_INPUT_READY | (dq.DQ_FLAG_OUTPUT_FREE if w > 0 else 0)
            p = _params(case, q, flags)
            s["grads"].append(g.worker())
            s["params"].append(p)
            s["msgs"].append(dq.Message(*_message_buffers(n, p), dseed, w, kind, p))
        if op == "step":
            s["side"] = g.side() if case["side"] == "vector" else None
            s["out"] = torch.empty(n, device="cuda")
    elif op in ("decode", "wire"):
        s["msgs"] = []
        for w, (q, kind, dseed) in enumerate(workers):
            p = _params(case, q)
            pk, sc = _message_buffers(n, p)
            _encoder(kind)(g.worker(), dseed, w, STEP, p, pk, sc)
            s["msgs"].append(dq.Message(pk, sc, dseed, w, kind, p))
        if op == "decode":
            s["side"] = g.side() if case["side"] == "vector" else None
            s["out"] = torch.empty(n, device="cuda")
        else:
            bits = s["msgs"][0].params.bits
            s["hist"] = torch.empty(1 << bits, dtype=torch.int64, device="cuda")
            if case["quant"] == "dqsg2":
                s["radix"] = torch.empty(dq.ternary_bytes(n), dtype=torch.uint8, device="cuda")
                s["stream"] = torch.empty(dq.packed_words(n, 2), dtype=torch.int32, device="cuda")
    else:
        s["msgs"] = []
        for w, (q, kind, dseed) in enumerate(workers):
            p = _params(case, q)
            grad = g.worker()
            dev = _message_buffers(n, p)
            _encoder(kind)(grad, dseed, w, STEP, p, *dev)
            pinned = _message_buffers(n, p, pinned=True)
            for a, b in zip(pinned, dev):
                a.copy_(b)
            s["msgs"].append(dq.Message(*pinned, dseed, w, kind, p))
        # the worker that encodes from host memory is the last one
        s["grad"] = torch.empty(n, pin_memory=True)
        s["grad"].copy_(grad)
        s["sent"] = _message_buffers(n, p, pinned=True)
        s["out"] = torch.empty(n, pin_memory=True)
        s["enc_ws"] = torch.empty(dq.encode_workspace_bytes(n, p), dtype=torch.uint8, device="cuda")
        s["dec_ws"] = torch.empty(dq.decode_workspace_bytes(s["msgs"], n, False), dtype=torch.uint8, device="cuda")
    return s


# ------------------------------------------------------------------------------------------------------ one pass
def _decode(s):
    case, msgs, n = s["case"], s["msgs"], s["n"]
    if case["side"] == "running":
        return dq.ndqsg_decode_aggregate_running(msgs, n, STEP, s["out"])
    if case["side"] == "first":
        return dq.ndqsg_decode_aggregate_side_first(msgs, n, STEP, s["out"])
    if case["side"] == "none":
        return dq.dqsg_decode_aggregate(msgs, n, STEP, s["out"])
    return dq.ndqsg_decode_aggregate(msgs, n, STEP, s["side"], s["out"])


def run(s):
    op = s["op"]
    if op == "decode":
        return _decode(s)
    if op in ("encode", "step"):
        sent = []
        for grad, p, m in zip(s["grads"], s["params"], s["msgs"]):
            sent.append(_encoder(m.kind)(grad, m.seed, m.worker, STEP, p, m.packed, m.scale))
        return sent if op == "encode" else (sent, _decode(s))
    if op == "host":
        m = s["msgs"][-1]
        sent = dq.ndqsg_encode_host(s["grad"], m.seed, m.worker, STEP, m.params, *s["sent"], s["enc_ws"])
        return sent, dq.ndqsg_decode_aggregate_side_first_host(s["msgs"], s["n"], STEP, s["out"], s["dec_ws"])
    m = s["msgs"][0]
    hist = dq.code_histogram(m.packed, s["n"], m.params.bits, s["hist"])
    if "radix" not in s:
        return hist
    radix = dq.ternary_pack(m.packed, s["n"], s["radix"])
    return hist, radix, dq.ternary_unpack(radix, s["n"], s["stream"])


# ------------------------------------------------------------------------------------------------------ accounting
def work(case):
    """Bytes: gradients, messages, side information and means, each once.  Operations: a dither value is a quarter
    of a Philox4x32-10 block (ten rounds of two multiplies and four XORs for four values; an eighth of one with the
    16-bit stream), quantizing and packing about six, unpacking, resolving and accumulating about ten."""
    op, n, bucket = case["op"], case["n"], case["bucket"]
    dither = 15 if case["dither"] == 32 else 8
    msg = sum(4 * ((n * QUANT[q]["bits"] + 31) // 32) + 4 * (-(-n // bucket)) for q, _, _ in _workers(case))
    W = len(_workers(case))
    encode = {"bytes": 4 * n * W + msg, "flops": n * W * (dither + 6)}
    decode = {"bytes": msg + 4 * n * (2 if case.get("side") == "vector" else 1), "flops": n * W * (dither + 10)}
    if op == "encode":
        return encode
    if op == "decode":
        return decode
    if op == "step":
        return {k: encode[k] + decode[k] for k in encode}
    if op == "host":
        sent = msg - sum(4 * ((n * QUANT[q]["bits"] + 31) // 32) + 4 * (-(-n // bucket))
                         for q, _, _ in _workers(case)[:-1])
        return {"bytes": 4 * n + sent + msg + 4 * n, "flops": n * (dither + 6) + decode["flops"]}
    bits = QUANT[case["quant"]]["bits"]
    stream = 4 * ((n * bits + 31) // 32)
    if case["quant"] == "dqsg2":
        return {"bytes": 2 * stream + stream + 2 * ((n + 4) // 5), "flops": 5 * n}
    return {"bytes": stream, "flops": n}


def tolerance(case):
    """Messages, counts and containers are whole numbers and scales are maxima: exact.  A mean of at most 32 fp32
    reconstructions, each a few roundings from the real value, is good to about 1e-6."""
    if case["op"] in ("encode", "wire"):
        return "exact"
    return {"rel": 2e-6, "max": 2e-5, "differ": 0.0}
