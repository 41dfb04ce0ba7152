"""The trace's per-thread work counters (csrc/work_count.cuh), compiled for the host:
no 32-bit sum wraps, however many crossings one packet makes before its end, and the
rule for the runs in which one could."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <stdio.h>
#include <stdlib.h>
#include "work_count.cuh"
int main(int argc, char** argv) {
    // traversals of up to argv[1] crossings, argv[2] of them in one packet
    const unsigned top = (unsigned)strtoul(argv[1], 0, 10);
    unsigned c = 0, r = 12345;
    unsigned long long total = 0, want = 0;
    for (long k = 0; k < atol(argv[2]); ++k) {
        r = r * 1664525u + 1013904223u;
        const unsigned n = k % 3 ? r % (top + 1u) : top;
        want += n;
        if (skirt::count_add(c, n)) { total += c; c = 0; }
    }
    printf("%llu %llu\n", total + c, want);
    for (int k = 3; k + 2 < argc; k += 3)
        printf("%d\n", (int)skirt::counts_within_packet(atoi(argv[k]), atoi(argv[k + 1]), strtoull(argv[k + 2], 0, 10)));
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("count")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-O1", "-I", os.path.join(ROOT, "paper_1705_04702_gb300", "csrc"), "-o", str(d / "h"),
                    str(d / "h.cpp")], check=True)
    return lambda *a: subprocess.run([str(d / "h")] + [str(v) for v in a], check=True, capture_output=True,
                                     text=True).stdout.split()


@pytest.mark.parametrize("top,count", [(0, 5), (400, 20_000_000), (1 << 24, 2000), ((1 << 31) - 1, 1000),
                                       ((1 << 31) + (1 << 30) - 1, 1000)])
def test_no_sum_wraps(harness, top, count):
    got, want = (int(v) for v in harness(top, count))
    assert got == want and (count < 100 or top < 400 or want >= 1 << 32)


def test_runs_whose_packets_may_wrap_a_counter(harness):
    """Every run for which the largest count of one packet and what may stay from
    those before reach 2^32 is told apart; the default event cap on ordinary grids is
    not."""
    cases = [(ev, ins, line) for ev in (1, 100, 10_000, 670_000, 2 ** 31 - 1) for ins in (0, 3, 16)
             for line in (3, 776, 3 * 4096 + 8, 2 ** 24, 2 ** 31)]
    got = [int(v) for v in harness(0, 0, *[v for c in cases for v in c])[2:]]
    for (ev, ins, line), g in zip(cases, got):
        worst = (ev + 1) * (ins + 2) * line + 2 ** 30 - 1
        assert g or worst < 2 ** 32, (ev, ins, line)
        assert not g or worst > 2 ** 31, (ev, ins, line)
    assert not got[cases.index((10_000, 16, 776))] and got[cases.index((670_000, 16, 776))]
