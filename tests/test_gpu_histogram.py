"""The code histogram at the lengths where its kernels change (CTAs of the cluster, the grid-wide kernel) and at ragged
ends whose pad bits are not zero, against numpy's counts of the codes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from test_gpu_parity import dq  # noqa: E402,F401

CLUSTER_BITS = 8 * (3 << 19)            # longest message that one cluster counts


@pytest.mark.parametrize("bits", range(1, 9))
@pytest.mark.parametrize("n", [1, 5, 63, 64, 65, 8191, 8193, 65536 + 3, 300_001, "edge", "past"])
def test_histogram_counts(dq, bits, n):
    if n in ("edge", "past"):
        if bits > 2:
            pytest.skip("one kernel for all lengths")
        n = CLUSTER_BITS // bits + (1 if n == "past" else 0)
    words = np.random.default_rng(n + bits).integers(0, 1 << 32, size=-(-n * bits // 32), dtype=np.uint32)
    codes = np.unpackbits(words.view(np.uint8), bitorder="little")[:n * bits].reshape(n, bits)
    want = np.bincount(codes.astype(np.int64) @ (1 << np.arange(bits)), minlength=1 << bits)
    hist = torch.full((1 << bits,), -7, dtype=torch.int64, device="cuda")      # whatever was there is overwritten
    dq.code_histogram(torch.from_numpy(words.view(np.int32)).cuda(), n, bits, hist)
    assert np.array_equal(hist.cpu().numpy(), want)
