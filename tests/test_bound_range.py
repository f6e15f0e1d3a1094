"""The bins of the running bound's histogram (csrc/bound_bins.cuh) over all scores a query can have, compiled for the
host: up to its largest product bound times its number of terms, and down to the negative of that, two scores an
eighth apart never share a bin, so that the bound never gets coarser than 8 bins an octave. Floors and bins agree for
every number of terms."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <vector>
#include "bound_bins.cuh"
using namespace sindi;
static uint32_t order(float s) {
    s = s + 0.0f;
    uint32_t u;
    std::memcpy(&u, &s, 4);
    return u & 0x80000000u ? ~u : u | 0x80000000u;
}
int main(int argc, char** argv) {
    const int terms = std::atoi(argv[1]);
    const float M = (float)std::atof(argv[2]);
    const int32_t top = hbin_top(order(M), terms);
    auto bin = [&](float s) { return (int)hbin(order(s), top); };
    const float most = M * (float)terms;
    for (float s = most; s > most / 65536.0f; s /= 1.126f)  // 16 octaves
        if (bin(s) <= bin(s / 1.126f)) return std::printf("%g and %g share a bin\n", s, s / 1.126f), 1;
    // the negative side: 12 octaves under the bins' top, which holds at least eight terms
    for (float s = most; s > M * (float)std::max(terms, 8) / 4096.0f; s /= 1.126f)
        if (bin(-s) >= bin(-s / 1.126f)) return std::printf("%g and %g share a bin\n", -s, -s / 1.126f), 1;
    if (!(bin(-most / 65536.0f) < bin(0.0f) && bin(0.0f) < bin(most / 65536.0f) && bin(0.0f) == bin(-0.0f)))
        return std::printf("zero\n"), 1;
    for (int oct = 0; oct < 50; oct++)  // and no score down to 2^-50 of it ends up with the zeros
        if (bin(std::ldexp(most, -oct)) == bin(0.0f)) return std::printf("2^-%d\n", oct), 1;
    std::mt19937 rng(5);
    std::vector<uint32_t> ob = {0u, 1u, 0x7FFFFFFFu, 0x80000000u, 0x80000001u, 0xFF7FFFFFu, 0xFF800000u};
    for (int i = 0; i < 20000; i++) ob.push_back(rng() % 0xFF800000u);
    for (int b = 0; b < kHBins; b++) {
        const uint32_t f = hbin_floor((uint32_t)b, top);
        if (f && f <= 0xFF800000u) { ob.push_back(f); ob.push_back(f - 1); }
    }
    for (int b = 0; b < kHBins; b++) {
        const uint32_t f = hbin_floor((uint32_t)b, top);
        for (uint32_t x : ob)
            if ((hbin(x, top) >= (uint32_t)b) != (x >= f)) return std::printf("bin %d, bits %x\n", b, x), 1;
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    d = tmp_path_factory.mktemp("range")
    (d / "r.cpp").write_text(SRC)
    csrc = os.path.join(ROOT, "paper_2509_08395_gb300", "csrc")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I" + csrc, str(d / "r.cpp"), "-o", str(d / "r")])
    return str(d / "r")


@pytest.mark.parametrize("largest", ["1", "0.0371", "1e9", "1e-9", "1e-20"])
@pytest.mark.parametrize("terms", [1, 8, 9, 20, 100, 128, 129, 2048])
def test_no_score_a_query_can_have_shares_a_wide_bin(checker, terms, largest):
    subprocess.run([checker, str(terms), largest], check=True)
