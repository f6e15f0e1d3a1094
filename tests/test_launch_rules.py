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
