"""The rule for buffers kept from one use to the next, with an allocator that fails above a
limit: the recorded capacity is never more than what was allocated."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1912_08445_gb300", "csrc")
PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "kept.h"
int main(int argc, char **argv) {
    const int64_t limit = atoll(argv[1]);
    int64_t cap = 0, held = 0;
    for (int i = 2; i < argc; i++) {
        int calls = 0;
        const int rc = mg::kept_buffer(cap, atoll(argv[i]), [&](int64_t n) {
            calls++;
            held = 0;
            if (n > limit) return -5;
            held = n > 0 ? n : 1;
            return 0;
        });
        std::printf("%d %lld %lld %d\n", rc, (long long)cap, (long long)held, calls);
    }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("kept")
    (d / "p.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I" + CSRC, str(d / "p.cpp"), "-o", str(d / "p")], check=True)
    return str(d / "p")


def _run(program, limit, *counts):
    out = subprocess.run([program, str(limit), *map(str, counts)], capture_output=True, text=True, check=True).stdout
    return [tuple(map(int, line.split())) for line in out.splitlines()]


def test_room_to_spare_is_recorded_only_when_it_was_had(program):
    assert _run(program, 10**9, 100000) == [(0, 103125, 103125, 1)]
    assert _run(program, 101000, 100000) == [(0, 100000, 100000, 2)]     # no room for the 3 %
    # what then fits the 3 % but not the buffer is a new allocation, here one that fails
    assert _run(program, 101000, 100000, 102000) == [(0, 100000, 100000, 2), (-5, 0, 0, 2)]
    assert _run(program, 101000, 100000, 100900)[1] == (0, 100900, 100900, 2)


def test_reuse_growth_and_giving_back(program):
    runs = _run(program, 10**9, 100000, 103125, 60000, 103126, 40000, 0, 1)
    assert runs[0] == (0, 103125, 103125, 1)
    assert runs[1] == (0, 103125, 103125, 0) and runs[2] == (0, 103125, 103125, 0)   # reused
    assert runs[3] == (0, 106348, 106348, 1)                                         # too small
    assert runs[4] == (0, 41250, 41250, 1)                                           # more than half empty
    assert runs[5] == (0, 1, 1, 1) and runs[6] == (0, 1, 1, 0)
