"""Passes of the stable counting sort, for every size that its callers may bring: up to 2^31 - 1
items and keys.  The planner is host arithmetic (partition.h); it is compiled here, and the passes
that it lays out are carried out in numpy."""
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1910_13555_gb300", "csrc")
MAIN = r"""
#include <cstdio>
#include "partition.h"
int main() {
  long long n, k;
  while (std::scanf("%lld %lld", &n, &k) == 2) {
    const bst::PartitionPlan P = bst::partition_plan(n, k);
    std::printf("%d %d", P.passes, P.bits);
    for (int i = 0; i < P.passes; ++i) std::printf(" %lld %lld", (long long)P.segment[i], (long long)P.keys[i]);
    std::printf("\n");
  }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("partition")
    (d / "m.cc").write_text(MAIN)
    exe = str(d / "m")
    subprocess.run(["g++", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover", "-I", CSRC,
                    str(d / "m.cc"), "-o", exe], check=True)

    def run(pairs):
        text = "".join(f"{n} {k}\n" for n, k in pairs)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, timeout=60, check=True)
        return [list(map(int, l.split())) for l in out.stdout.splitlines()]
    return run


EDGE = [1, 2, 255, 256, 257, 8192, 65535, 65536, 80000, 1 << 20, (1 << 24) - 1, 1 << 24, (1 << 24) + 1,
        17640000, 500000000, (1 << 30) - 1, 1 << 30, (1 << 30) + 1, (1 << 31) - 1]


def test_every_size_ends_within_the_cells(plan):
    pairs = [(n, k) for n in EDGE for k in EDGE]
    for (n, k), (passes, bits, *rest) in zip(pairs, plan(pairs), strict=True):
        covered = 0
        for segment, keys in zip(rest[::2], rest[1::2], strict=True):
            assert segment >= 256 and keys >= 1
            assert keys * -(-n // segment) <= 1 << 24
            covered += bits
        assert passes == len(rest) // 2 and (passes == 1 or 1 << covered >= k)


def test_the_former_sizes_keep_their_passes(plan):
    # one pass of segments of 256 and 512; two of the 2000 x 2000 banded plan's groups
    assert plan([(3_000_000, 1000)]) == [[1, 31, 256, 1000]]
    assert plan([(3_000_000, 2000)]) == [[1, 31, 512, 2000]]
    assert plan([(3_200_000, 80_000)]) == [[2, 9, 1024, 512, 1024, 157]]


@pytest.mark.parametrize("n,nkeys", [(4200, 17_640_000), (300, (1 << 31) - 1), (5000, 1 << 30),
                                     (20000, 9_000_001)])
def test_passes_sort_stably(plan, n, nkeys):
    rng = np.random.default_rng(n)
    keys = rng.integers(0, nkeys, n) if n != 5000 else rng.integers(nkeys - 7, nkeys, n)
    (passes, bits, *rest), = plan([(n, nkeys)])
    assert passes > 1
    perm = np.arange(n)
    for i in range(passes):
        digit = keys[perm] >> (i * bits)
        if i + 1 < passes:
            digit &= (1 << bits) - 1
        assert digit.max() < rest[2 * i + 1]
        perm = perm[np.argsort(digit, kind="stable")]
    assert (perm == np.argsort(keys, kind="stable")).all()
