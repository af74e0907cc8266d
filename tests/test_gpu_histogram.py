"""The code histogram at the lengths where its kernels change (CTAs of the cluster, the grid-wide kernel) and at ragged
ends whose pad bits are not zero, against numpy's counts of the codes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from test_gpu_parity import dq  # noqa: E402,F401

CLUSTER_BITS = 8 * (3 << 19)            # longest message that one cluster counts


def _counts(words, n, bits):
    out = np.zeros(1 << bits, dtype=np.int64)
    for lo in range(0, n, 1 << 23):                 # (a piece of codes starts at a word)
        hi = min(n, lo + (1 << 23))
        b = np.unpackbits(words[lo * bits // 32:-(-hi * bits // 32)].view(np.uint8), bitorder="little")
        codes = b[:(hi - lo) * bits].reshape(hi - lo, bits) @ (1 << np.arange(bits)).astype(np.uint8)
        out += np.bincount(codes, minlength=1 << bits)
    return out


@pytest.mark.parametrize("bits", range(1, 9))
@pytest.mark.parametrize("n", [1, 5, 63, 64, 65, 8191, 8193, 65536 + 3, 300_001, "edge", "past"])
def test_histogram_counts(dq, bits, n):
    if n in ("edge", "past"):
        if bits > 2:
            pytest.skip("one kernel for all lengths")
        n = CLUSTER_BITS // bits + (1 if n == "past" else 0)
    words = np.random.default_rng(n + bits).integers(0, 1 << 32, size=-(-n * bits // 32), dtype=np.uint32)
    want = _counts(words, n, bits)
    hist = torch.full((1 << bits,), -7, dtype=torch.int64, device="cuda")      # whatever was there is overwritten
    dq.code_histogram(torch.from_numpy(words.view(np.int32)).cuda(), n, bits, hist)
    assert np.array_equal(hist.cpu().numpy(), want)


@pytest.mark.parametrize("bits", [3, 4, 5])
@pytest.mark.parametrize("n", [79_999_999, 80_000_003])      # the last with counters per warp, one with counters per thread
def test_histogram_counts_of_very_long_messages(dq, bits, n):
    words = np.random.default_rng(n + bits).integers(0, 1 << 32, size=-(-n * bits // 32), dtype=np.uint32)
    hist = dq.code_histogram(torch.from_numpy(words.view(np.int32)).cuda(), n, bits)
    assert np.array_equal(hist.cpu().numpy(), _counts(words, n, bits))


@pytest.mark.parametrize("bits", range(1, 9))
def test_histogram_of_one_code_only(dq, bits):
    n, code = 2_000_003, (1 << bits) - 1
    words = torch.full((-(-n * bits // 32),), -1, dtype=torch.int32, device="cuda")
    want = torch.zeros(1 << bits, dtype=torch.int64)
    want[code] = n
    assert torch.equal(dq.code_histogram(words, n, bits).cpu(), want)
