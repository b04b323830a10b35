"""The packed counter of new partial matches (rows << 40 | sum of fan-outs): warps
look at it, add and test what they found, many at a time. Whatever the order, rows
that were given out stay below the first one that found no room, unless the sum of
fan-outs ran out, which every such run must notice."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "common.cuh"
using namespace gfd;
int main(int, char** a) {  // warps in flight, partial matches, fan-out of each, rows there is room for
    const uint64_t warps = atoll(a[1]), fo = atoll(a[3]), cap = atoll(a[4]);
    uint64_t left = atoll(a[2]), ctr = 0, limit = ~0ull, stored = 0, in_place = 0, top = 0;
    const uint64_t all = left, add = (32ull << ROW_SHIFT) + 32 * fo;
    bool ended = false;
    while (left) {
        std::vector<int> look;
        for (uint64_t w = 0; w < warps && left; w++, left -= std::min<uint64_t>(left, 32))
            look.push_back(counter_add(ctr, add, cap));
        for (int full : look) {
            uint64_t old = 0;
            if (full == ROWS_FIT) {
                old = ctr;
                ctr += add;
                full = counter_add(old, add, cap);
                if (full == ROWS_OUT) limit = std::min(limit, old);
            }
            ended |= full == WORK_OUT;
            if (full == ROWS_OUT) in_place += 32;
            if (full == ROWS_FIT) stored += 32, top = std::max(top, old);
        }
    }
    if (ended) return puts("ended"), 0;
    const bool kept = stored == 0 || top < limit;
    printf("%s\n", kept && stored + in_place == all && std::min(ctr, limit) >> ROW_SHIFT == stored ? "all" : "lost");
}
"""


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    d = tmp_path_factory.mktemp("counter")
    (d / "m.cpp").write_text(PROGRAM)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2608_02321_gb300", "csrc"), "-I",
                    os.path.join(cuda, "include"), str(d / "m.cpp"), "-o", str(d / "m")], check=True)
    return str(d / "m")


@pytest.mark.parametrize("warps", [1, 8, 9728])
@pytest.mark.parametrize("n,fanout,cap,want", [
    (1_000_000, 1_000_000, 15_000_000, "all"),     # a sum just below 2^40
    (2_000_000, 1_000_000, 15_000_000, "ended"),   # beyond it
    (1_000_000, 100, 4_096, "all"),                # rows run out
    (1_000_000, 1_000_000, 500_000, "all"),        # rows run out below 2^40, the rest passes it in place
    (64_000, 1 << 31, 15_000_000, "ended"),        # the longest lists
])
def test_every_partial_match_is_kept_or_the_slot_ends(model, warps, n, fanout, cap, want):
    out = subprocess.run([model, str(warps), str(n), str(fanout), str(cap)], check=True, capture_output=True, text=True)
    assert out.stdout.strip() == want
