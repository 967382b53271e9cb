"""Tiles of a batch's scan: every tile of every instance has one block, and the
number of blocks grows with the rows of the batch, not with its largest
instance times its count (compiled from the library's header, no GPU)."""
import os
import shutil
import subprocess
import textwrap

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_11988_gb300", "csrc")

PROGRAM = textwrap.dedent(r"""
    #include <cstdio>
    #include <vector>
    #include "queues.h"
    using namespace ts;
    // reads: chunk offset of the first instance, their number, their rows; prints the blocks, then (instance,
    // tile) of each block that has rows or is its instance's first
    int main() {
        long long c, count;
        if (scanf("%lld %lld", &c, &count) != 2) return 1;
        std::vector<long long> off, rows(count);
        for (auto& n : rows) {
            if (scanf("%lld", &n) != 1) return 1;
            off.push_back(c);
            c += (n + 31) / 32;
        }
        const long long blocks = bat_tile_span(off[0], off[count - 1], (int)count, rows[count - 1]);
        printf("%lld\n", blocks);
        for (long long x = 0; x < blocks; ++x) {
            const long long at = bat_first_tile(off[0], 0) + x;
            const int b = bat_inst_of_tile([&](int k) { return off[k]; }, (int)count, at);
            const long long tile = at - bat_first_tile(off[b], b);
            if (tile == 0 || tile * BAT_TILE < rows[b]) printf("%d %lld\n", b, tile);
        }
        return 0;
    }
""")


@pytest.fixture(scope="module")
def tiles(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("tiles")
    src, exe = d / "t.cpp", d / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)

    def run(first, rows):
        out = subprocess.run([str(exe)], input=" ".join(map(str, [first, len(rows), *rows])), capture_output=True,
                             text=True, check=True).stdout.split("\n")
        return int(out[0]), [tuple(map(int, x.split())) for x in out[1:] if x]

    return run


def _batches():
    rng = np.random.default_rng(0)
    yield 0, [0]
    yield 0, [1]
    yield 5, [4095, 4096, 4097, 0, 0, 8192, 8193, 1, 0]
    yield 130, [300000] + [50] * 3000
    yield 7, [50] * 3000 + [300000]
    for _ in range(30):
        k = int(rng.integers(1, 200))
        yield int(rng.integers(0, 10000)), [int(x) for x in rng.integers(0, rng.choice([3, 5000, 40000]), k)]


def test_every_tile_once_and_few_blocks(tiles):
    for first, rows in _batches():
        blocks, seen = tiles(first, rows)
        want = [(b, t) for b, n in enumerate(rows) for t in range(max(1, -(-n // 4096)))]
        assert seen == want
        assert blocks <= sum(rows) // 4096 + 2 * len(rows) + 1
