"""The work queue's refill (csrc/queue_chunk.cuh), compiled for the host: a refill that
the caller names is taken to the letter at every size, and the default is the
largest of 1 to 4 that leaves every thread eight refills."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <stdio.h>
#include <stdlib.h>
#include "queue_chunk.cuh"
int main(int argc, char** argv) {
    for (int k = 1; k + 2 < argc; k += 3)
        printf("%d\n", skirt::queue_chunk(atoi(argv[k]), strtoull(argv[k + 1], 0, 10), strtoull(argv[k + 2], 0, 10)));
}
"""


@pytest.fixture(scope="module")
def chunk(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("chunk")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-O1", "-I", os.path.join(ROOT, "paper_1705_04702_gb300", "csrc"), "-o", str(d / "h"),
                    str(d / "h.cpp")], check=True)

    def call(cases):
        out = subprocess.run([str(d / "h")] + [str(v) for c in cases for v in c], check=True, capture_output=True, text=True)
        return [int(v) for v in out.stdout.split()]

    return call


def test_a_named_refill_is_taken_to_the_letter(chunk):
    cases = [(c, n, t) for c in (1, 3, 4, 16, 1 << 20) for n in (0, 1, 500, 100_000, 10 ** 12) for t in (64, 116_736)]
    assert chunk(cases) == [c for c, _, _ in cases]


def test_default_leaves_eight_refills(chunk):
    t = 116_736
    cases = [(0, n, t) for n in (0, 1, 8 * t - 1, 8 * t, 16 * t - 1, 16 * t, 24 * t, 32 * t - 1, 32 * t, 10 ** 12)]
    assert chunk(cases) == [1, 1, 1, 1, 1, 2, 3, 3, 4, 4]
    assert chunk([(0, 2 ** 63, 1), (0, 5, 0)]) == [4, 1]
