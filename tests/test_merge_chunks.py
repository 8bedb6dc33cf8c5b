"""The chunks of the merge-path product, on the CPU: every entry of a range is in
one chunk and every row that ends in the range is flagged in the chunk that holds
its last entry, also where the entries end just below 2^31."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_02530_gb300", "csrc")

PROGRAM = r"""
#include "merge_chunks.h"
#include <cstdlib>
using namespace spmvk;
int main(int argc, char** argv) {   // rows of `len` entries, the range [k1 - n, k1)
    const int k1 = std::atoi(argv[1]), n = std::atoi(argv[2]), len = std::atoi(argv[3]), k0 = k1 - n;
    long long seen = 0, chunks = 0, rows = 0, flagged = 0;
    const long long end = (long long)k0 + len / 2 + 1;   // the first row begins before the range
    for (long long e = end; e <= k1; e += len) ++rows;
    long long next = end;
    for (unsigned c = merge_first_chunk(k0); c < (unsigned)k1; c += MERGE_CHUNK) {
        if (++chunks > n / MERGE_CHUNK + 2) return 1;
        for (unsigned e = c; e != c + MERGE_CHUNK; ++e) seen += merge_in_range(e, k0, k1);
        for (; next <= k1 && merge_ends_by((int)next, c); next += len) {
            if ((unsigned)next - 1 - c >= (unsigned)MERGE_CHUNK) return 2;   // the flag's place
            ++flagged;
        }
    }
    return seen != n ? 3 : flagged != rows ? 4 : 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("chunks")
    (d / "c.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-ftrapv", "-I", CSRC, str(d / "c.cpp"), "-o", str(d / "c")], check=True)
    return str(d / "c")


@pytest.mark.parametrize("k1", [600, 2**20 + 3, 2**31 - 320, 2**31 - 256, 2**31 - 72, 2**31 - 65])
@pytest.mark.parametrize("n", [1, 7, 8, 248, 249, 504])
@pytest.mark.parametrize("length", [1, 3, 8, 100, 1000])
def test_chunks_hold_the_range(program, k1, n, length):
    assert subprocess.run([program, str(k1), str(n), str(length)]).returncode == 0
