"""How much memory a search asks for (csrc/launch_rules.cuh), compiled for the host and run against a device that is
made up: an allocation succeeds while it fits the free bytes."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "launch_rules.cuh"
using namespace sindi;
int main(int argc, char** argv) {
    const long long a = std::atoll(argv[2]), b = std::atoll(argv[3]);
    if (!std::strcmp(argv[1], "fits")) {  // a queries, b of which there is room for
        long long tries = 0;
        const long long got = largest_that_fits(a, [&](int64_t c) { tries++; return c <= b; });
        std::printf("%lld %lld\n", got, tries);
    } else {  // a windows, b queries, bytes a chain
        std::printf("%d 0\n", graph_lanes((uint32_t)a, b, (size_t)std::atoll(argv[4])));
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "r.cpp").write_text(SRC)
    csrc = os.path.join(ROOT, "paper_2509_08395_gb300", "csrc")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I" + csrc, str(d / "r.cpp"), "-o", str(d / "r")])
    return lambda *a: [int(x) for x in subprocess.check_output([str(d / "r"), *map(str, a)]).split()]


@pytest.mark.parametrize("n", [1, 2, 3, 5, 1000, 65535])
def test_a_batch_takes_the_largest_group_there_is_room_for(run, n):
    for room in (0, 1, 2, n // 4, n // 2, n - 1, n, n + 1):
        got, tries = run("fits", n, room)
        assert tries <= n.bit_length() + 1
        if room == 0:
            assert got == 0
        elif room >= n:
            assert (got, tries) == (n, 1)
        else:  # a group of more than half of what fits, and never less than one query
            assert 1 <= got <= room and 2 * got >= room


MIB = 1 << 20


@pytest.mark.parametrize("sigma", [1, 7, 8, 62, 1075])
@pytest.mark.parametrize("queries", [2, 23, 100, 119, 120, 200, 1000, 100_000])
@pytest.mark.parametrize("lane_bytes", [100_000, 512 * 1024, 17 * MIB, 21 * MIB, 22 * MIB, 141 * MIB, 4096 * MIB])
def test_more_chains_only_while_their_workspaces_are_small(run, sigma, queries, lane_bytes):
    lanes, _ = run("lanes", sigma, queries, lane_bytes)
    assert 1 <= lanes <= min(56, queries)
    assert lanes >= min(24, queries)  # what direct launches use
    assert lanes <= 24 or lanes * lane_bytes <= 512 * MIB
    if sigma < 8 or queries <= 120 or lane_bytes >= 22 * MIB:
        assert lanes == min(24, queries)
    if sigma >= 8 and queries >= 280 and lane_bytes <= 9 * MIB:
        assert lanes == 56
