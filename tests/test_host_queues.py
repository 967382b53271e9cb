"""Queues of rows cut into chunks: every chunk of the longest row a matrix can
have (2^31 - 1 columns) has a number of its own, with the packing and the chunk
lengths that the sources use (host arithmetic, no GPU)."""
import os
import re
import shutil
import subprocess
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2408_11988_gb300", "csrc")
LONGEST = 2**31 - 1

PROGRAM = textwrap.dedent(r"""
    #include <cstdio>
    #include "queues.h"
    using namespace ts;
    int main() {
        long long r, c;
        while (scanf("%lld %lld", &r, &c) == 2) {
            const long long x = queue_item(r, c);
            printf("%d %lld %lld\n", x >= 0, item_row(x), item_chunk(x));
        }
        return 0;
    }
""")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def constant(name, text):
    return int(re.search(r"constexpr int %s = (\d+)" % name, text).group(1))


@pytest.mark.parametrize("name,chunk,extra", [("force2vec.cu", "F2V_CHUNK", 32), ("msbfs.cu", "BFS_CHUNK", 0),
                                              ("batched.cu", "PREP_LONG", 0), ("spgemm.cu", "LONG_CHUNK", 0)])
def test_chunks_of_the_longest_row_are_numbered(name, chunk, extra):
    text = source(name)
    shifts = {int(x) for x in re.findall(r"items\[[^\]]*\] >> (\d+)|item >> (\d+)", text) for x in x if x}
    bits = min(shifts) if shifts else 32  # queue_item
    assert shifts or "queue_item(" in text
    chunks = -(-(LONGEST + extra) // constant(chunk, text))
    assert chunks <= 2**bits, (name, chunks, bits)


def test_queue_items_round_trip(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "q.cpp", tmp_path / "q"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    chunks = -(-(LONGEST + 32) // constant("F2V_CHUNK", source("force2vec.cu")))
    pairs = [(r, c) for r in (0, 1, 12345, LONGEST) for c in (0, 1, 2**24 - 1, 2**24, 2**24 + 5, chunks - 1)]
    out = subprocess.run([str(exe)], input="\n".join("%d %d" % p for p in pairs), capture_output=True, text=True,
                         check=True).stdout.split("\n")
    assert [tuple(map(int, x.split())) for x in out if x] == [(1, r, c) for r, c in pairs]


def test_batched_long_rows_count_their_parts():
    # one 64-bit word per row: the products added so far below bit LONG_SHIFT,
    # the parts finished above it; neither may run into the other or out of the
    # word for the longest row over rows of B of 1024 entries
    text = source("batched.cu")
    part, shift = constant("PREP_LONG", text), constant("LONG_SHIFT", text)
    parts, products = -(-LONGEST // part), LONGEST * 1024
    assert products < 2**shift
    word = (parts << shift) + products
    assert word < 2**64
    assert (word >> shift, word & (2**shift - 1)) == (parts, products)
