"""The bins of the running bound's histogram (csrc/bound_bins.cuh), compiled for the host: for every bin, a score lies
in it or above exactly when its order bits reach the bin's floor; hbin never falls as the score grows."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <algorithm>
#include <cstdio>
#include <random>
#include <vector>
#include "bound_bins.cuh"
using namespace sindi;
int main(int argc, char** argv) {
    std::mt19937 rng(3);
    const uint32_t last = 0xFF800000u;  // the order bits of +inf
    const uint32_t m = (uint32_t)std::stoul(argv[1], nullptr, 0);
    const int32_t top = hbin_top(m);
    std::vector<uint32_t> ob = {0u, 1u, 0x7FFFFFFFu, 0x80000000u, 0x80000001u, last - 1, last};
    for (int i = 0; i < 40000; i++) ob.push_back(rng() % last);
    for (int b = 0; b < kHBins; b++) {
        const uint32_t f = hbin_floor((uint32_t)b, top);
        if (f && f <= last) { ob.push_back(f); ob.push_back(f - 1); }
    }
    std::sort(ob.begin(), ob.end());
    for (size_t i = 1; i < ob.size(); i++)
        if (hbin(ob[i], top) < hbin(ob[i - 1], top)) return std::printf("hbin falls\n"), 1;
    for (int b = 0; b < kHBins; b++) {
        const uint32_t f = hbin_floor((uint32_t)b, top);
        for (uint32_t x : ob)
            if ((hbin(x, top) >= (uint32_t)b) != (x >= f)) return std::printf("bin %d, bits %x\n", b, x), 1;
    }
    // the fine range: bins of 2^-6 of an octave, from three octaves above M down
    if (m >= 0xA0000000u && m < 0xE0000000u) {
        for (int b = kHBins - kHFine; b + 1 < kHBins; b++)
            if (hbin_floor(b + 1, top) - hbin_floor(b, top) != 1u << 17) return std::printf("bin width\n"), 1;
        if (hbin(m, top) != (uint32_t)(kHBins - 1 - 3 * 64)) return std::printf("M's bin\n"), 1;
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    d = tmp_path_factory.mktemp("bins")
    (d / "bins.cpp").write_text(SRC)
    csrc = os.path.join(ROOT, "paper_2509_08395_gb300", "csrc")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I" + csrc, str(d / "bins.cpp"), "-o", str(d / "bins")])
    return str(d / "bins")


@pytest.mark.parametrize("order_bits", [0x80000000, 0x80000001, 0x80800000, 0x9F000000, 0xBF800000, 0xC1234567,
                                        0xFF000000, 0xFF7FFFFF, 0xFF800000, 0xFFFFFFFF],
                         ids=["zero", "tiniest", "least-normal", "small", "one", "ten", "huge", "largest", "inf", "nan"])
def test_bins_and_floors_agree(checker, order_bits):
    subprocess.run([checker, hex(order_bits)], check=True)
