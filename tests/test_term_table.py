"""The number of terms a term table takes from a query row (csrc/checks.cuh, table_terms), compiled for the host: it
counts entries of the arrays the table's kernel indexes, so it stays in 0 .. block for any row, also one whose offsets
decrease (device offsets are not checked before a search)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2509_08395_gb300", "csrc")

SRC = r"""
#include <climits>
#include <initializer_list>
#include <cstdio>
#include <cstdlib>
#include "checks.cuh"
int main(int argc, char** argv) {
    const int block = std::atoi(argv[1]);
    for (int nt : {INT_MIN, INT_MIN + 1, -100000, -1, 0, 1, block - 1, block, block + 1, 3 * block + 5, 2048}) {
        int taken = 0;
        for (int c0 = 0; c0 == 0 || c0 < nt; c0 += block) {  // the scan's loop over tables
            const int nc = sindi::table_terms(nt, c0, block);
            if (nc < 0 || nc > block) return std::printf("nt %d c0 %d: %d\n", nt, c0, nc), 1;
            taken += nc;
        }
        if (taken != (nt > 0 ? nt : 0)) return std::printf("nt %d: %d terms taken\n", nt, taken), 1;
    }
    return 0;
}
"""


@pytest.mark.parametrize("block", [128, 224, 256, 384, 512, 1024])
def test_table_terms(tmp_path, block):
    (tmp_path / "t.cpp").write_text(SRC)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I" + CSRC, str(tmp_path / "t.cpp"), "-o", str(tmp_path / "t")])
    subprocess.run([str(tmp_path / "t"), str(block)], check=True)


def test_the_scan_takes_its_counts_from_it():
    src = open(os.path.join(CSRC, "search.cu")).read()
    assert "table_terms(nt, c0, kTermChunk)" in src
