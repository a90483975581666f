"""The sort kernels' ranges of slots at the largest plans (2^31 - 2 particles),
computed by the functions the kernels use, compiled for the host: no step of a
loop over a range leaves int32, and no slot is left out or read past the end."""
import os
import subprocess

import pytest

from paper_2003_11468_gb300 import build

MAX = 2147483646
SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "fof_internal.cuh"
int main(int, char** argv)
{
    const int first = atoi(argv[1]), count = atoi(argv[2]), of = atoi(argv[3]);
    for (int rank = 0; rank < of; ++rank) {
        const fofgpu::SlotRange r = fofgpu::slot_share(first, count, rank, of);
        printf("%d %d\n", r.first, r.count);
    }
    for (int k : {0, 1, 255, 511, 512, 2147483647})
        printf("%d %d\n", k, (int)fofgpu::slot_before(first, k, first + count));
}
"""


@pytest.fixture(scope="module")
def ranges(tmp_path_factory):
    d = tmp_path_factory.mktemp("slots")
    src, exe = str(d / "slots.cu"), str(d / "slots")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build.nvcc(), "-std=c++17", "-O1", "-I", build.CSRC, "-I", build.INCLUDE, *build.ARCH, src, "-o", exe],
                   check=True, capture_output=True)

    def run(first, count, of=8):
        out = subprocess.run([exe, str(first), str(count), str(of)], check=True, capture_output=True, text=True).stdout
        rows = [tuple(map(int, line.split())) for line in out.splitlines()]
        return rows[:of], rows[of:]

    yield run
    os.remove(exe)


STEP = 4 * 512                                # particles a CTA of the cluster steps by


@pytest.mark.parametrize("count", [0, 1, 7, 8, 9, 511, 8193, 100_000, 1 << 30, MAX - 3, MAX])
@pytest.mark.parametrize("room", [0, 1, 300, 5000])
def test_ranges_at_the_last_slots(ranges, count, room):
    first = max(MAX - count - room, 0)
    shares, before = ranges(first, count)
    at = first
    for start, n in shares:                   # in order, without gaps or overlap
        assert n >= 0 and (n == 0 or start == at)
        at += n
        assert n + STEP < 2 ** 31
    assert at == first + count
    for k, inside in before:
        assert inside == (k < count)
