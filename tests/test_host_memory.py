"""Which host buffers the kernels may work on without a copy (csrc/dq_host_memory.h): decided on the CPU, with made-up
page-locked ranges in the place of the driver's."""
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_1904_01197_b200" / "csrc"

# Allocation [4096, 4096 + 65536) at the same device address; registration [200000, 200000 + 10000) at 1 << 40;
# two registrations that touch, [1 << 20, + 4096) and [(1 << 20) + 4096, + 4096).
PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "dq_host_memory.h"

int main(int argc, char** argv)
{
    const uint64_t device[] = {4096, 1ull << 40, 1ull << 20, (1ull << 20) + 4096}, start[] = {4096, 200000, 1 << 20, (1 << 20) + 4096},
                   size[] = {65536, 10000, 4096, 4096};
    auto look = [&](const void* p, dq::PinnedRange* r) {
        const uint64_t a = (uint64_t)(uintptr_t)p;
        for (int i = 0; i < 4; ++i)
            if (a >= start[i] && a < start[i] + size[i]) {
                *r = {device[i] + (a - start[i]), start[i], size[i]};
                return true;
            }
        return false;
    };
    for (int i = 1; i + 1 < argc; i += 2)
        printf("%llu\n", (unsigned long long)dq::pinned_device_address((const void*)(uintptr_t)strtoull(argv[i], 0, 10),
                                                                      strtoull(argv[i + 1], 0, 10), look));
}
"""

CASES = [                                   # address, bytes, device address or 0
    (4096, 65536, 4096), (4096, 1, 4096), (4096 + 16, 65536 - 16, 4096 + 16), (4096 + 65520, 16, 4096 + 65520),
    (4096, 65537, 0),                       # one byte past the allocation
    (4096 + 16, 65536, 0), (4096 + 65520, 17, 0),
    (4096, 1 << 63, 0), (4096 + 16, (1 << 64) - 16, 0),                     # lengths that would wrap around
    (4096 + 4, 16, 0),                      # misaligned
    (200000, 10000, 1 << 40), (200016, 9984, (1 << 40) + 16), (200000, 10001, 0), (200000 + 9999, 1, 0),
    (100, 16, 0), (300000, 16, 0), (0, 16, 0),                              # not page-locked
    (1 << 20, 4096, 1 << 20), (1 << 20, 4112, 0),                           # across two registrations
]


@pytest.fixture(scope="module")
def decide(tmp_path_factory):
    d = tmp_path_factory.mktemp("host_memory")
    (d / "p.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", f"-I{CSRC}", "-o", str(d / "p"), str(d / "p.cpp")], check=True)
    return lambda cases: [int(v) for v in subprocess.run(
        [str(d / "p"), *[str(x) for c in cases for x in c[:2]]], check=True, capture_output=True, text=True).stdout.split()]


def test_only_buffers_that_are_page_locked_to_their_last_byte_are_used_in_place(decide):
    assert decide(CASES) == [c[2] for c in CASES]
