"""The pieces of a long row of the batched products, on the CPU: they cover the
row's entries once, in order, also where the row ends just below 2^31 entries
(the largest matrix a batch takes has 2^31 - 9)."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_02530_gb300", "csrc")

PROGRAM = r"""
#include "pieces.h"
#include <cstdio>
#include <cstdlib>
int main(int argc, char** argv) {
    const int len = std::atoi(argv[1]), L = std::atoi(argv[2]);
    const int n = spmvk::piece_count(len, L);
    long long next = 0;
    for (int p = 0; p < n; ++p) {
        const int size = spmvk::piece_size(len, L, p);
        if (size < 1 || size > L || next != (long long)p * L) return 1;
        next += size;
    }
    std::printf("%d %lld", n, next);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("pieces")
    (d / "p.cpp").write_text(PROGRAM)
    # signed overflow in the functions under test ends the program
    subprocess.run(["g++", "-std=c++17", "-O1", "-ftrapv", "-I", CSRC, str(d / "p.cpp"), "-o", str(d / "p")], check=True)
    return str(d / "p")


@pytest.mark.parametrize("piece_len", [512, 1024, 2048])
@pytest.mark.parametrize("length", [513, 2049, 4096, 2**31 - 2048, 2**31 - 513, 2**31 - 512, 2**31 - 10, 2**31 - 9])
def test_pieces_cover_the_row(program, length, piece_len):
    r = subprocess.run([program, str(length), str(piece_len)], capture_output=True, text=True)
    assert r.returncode == 0
    assert r.stdout == "%d %d" % (-(-length // piece_len), length)
