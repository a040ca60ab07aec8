"""How a tile of the staged FP64 kernel sums its outputs (fp64_tiles.h, compiled here for the host):
the splits fit the accumulators and the slot, the words hold them, and where a whole-tile split would
pay by the wide shape's accumulators no chosen form has longer chains than that split, unless none in
the tile's shape is shorter."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1910_13555_gb300", "csrc")
MAIN = r"""
#include <cstdio>
#include "fp64_tiles.h"
using namespace bst;
int main() {
  int mn, smax, tile, slot, whole, ne;
  while (std::scanf("%d %d %d %d %d %d", &mn, &smax, &tile, &slot, &whole, &ne) == 6) {
    TailCost tc = tail_cost(mn, smax);
    SplitSteps<unsigned> st;
    for (int e = 0; e < ne; ++e) {
      int w;
      if (std::scanf("%d", &w) != 1) return 1;
      tail_add(tc, w);
      st.add(w);
    }
    const TileChoice R = choose_tile(tc, st, mn, ne, smax, tile, slot, whole != 0);
    std::printf("%d %d %d %d %d %lld %lld %lld\n", R.split, R.tail, R.fresh, R.tail_fresh, choice_word(R),
                R.reference, R.unsplit, R.plain);
  }
}
"""


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("tiles")
    (d / "m.cu").write_text(MAIN)
    exe = str(d / "m")
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", CSRC, str(d / "m.cu"), "-o", exe], check=True, capture_output=True)

    def run(tiles):
        text = "".join(" ".join(map(str, (mn, smax, tile, slot, int(whole), len(w), *w))) + "\n"
                       for mn, smax, tile, slot, whole, w in tiles)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, timeout=120, check=True)
        return [list(map(int, l.split())) for l in out.stdout.splitlines()]
    return run


def _chains(mn, w, split, tail, fresh, tail_fresh):
    """Length of the longest chain of additions behind an output, as the rounding model counts it."""
    w1, ne = sum(w), len(w)
    if split > 1:
        return w1 // split + split
    width = -(-w1 // ne)
    long = 0
    if (mn >= 32 if tail > 1 else True):
        long = width + ne if fresh else w1
    if tail > 1:
        long = max(long, -(-width // tail) + ne if tail_fresh else w1 // tail + tail)
    return long


def test_choices_fit_and_keep_the_reference(choose):
    rng = np.random.default_rng(1)
    tiles = []
    for _ in range(4000):
        wide = rng.random() < 0.3
        tile, most = (544, 1184) if wide else (320, 896)
        mn = int(rng.integers(1, tile + 1)) if rng.random() < 0.5 else int(rng.choice([25, 49, 65, 81, 100, 115, 144, 169]))
        ne = int(rng.choice([1, 2, 3, 5, 9, 20, 60]))
        top = int(rng.choice([1, 4, 5, 13, 35, 60]))
        w = [int(x) for x in rng.integers(max(1, top // 2), top + 1, ne)]
        slot = int(rng.integers(max(mn, max(w)), most + 1)) if mn < most else most
        tiles.append((mn, int(rng.choice([1, 2, 4, 16])), tile, slot, bool(rng.random() < 0.7), w))
    paid = 0
    for (mn, smax, tile, slot, whole, w), got in zip(tiles, choose(tiles), strict=True):
        split, tail, fresh, tail_fresh, word, reference, unsplit, plain = got
        assert 1 <= split <= min(16, max(smax, 1)) and split * mn <= max(mn, min(tile, slot))
        assert 1 <= tail <= max(1, min(16, smax)) and (tail == 1 or tail * (mn % 32) <= 32)
        assert word == split | tail << 8 | fresh << 16 | tail_fresh << 17
        assert plain <= unsplit
        if reference == 0:
            continue
        paid += 1
        cost = lambda s: -(-s * mn // 32) * sum(-(-x // s) for x in w) + (s - 1) * -(-mn // 32)
        room = min(16, smax, min(544, slot) // mn)
        s0 = min(range(2, room + 1), key=cost)
        limit = sum(w) // s0 + s0
        mine = _chains(mn, w, split, tail, fresh, tail_fresh)
        if mine > limit:  # nothing shorter in this shape
            for s in range(2, min(16, smax, min(tile, slot) // mn) + 1):
                assert sum(w) // s + s >= mine
    assert paid > 200


def test_one_panel_and_no_split(choose):
    # a single panel; a bound of 1; outputs that fill their lanes
    for tile in [(65, 16, 320, 896, True, [49]), (65, 1, 320, 896, True, [35] * 60), (64, 16, 320, 896, True, [35] * 60)]:
        split, tail, fresh, tail_fresh, *_ = choose([tile])[0]
        if tile[1] == 1 or tile[0] == 64:
            assert (split, tail, tail_fresh) == (1, 1, 0)
