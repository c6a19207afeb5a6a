"""The counter of the weight table's pool of lines (csrc/pool.h), on the CPU: a sequence of claims
whose demands pass 2^32 lines many times over never gets a line twice and never lines beyond the
pool.  The same check finds out a 32-bit counter."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include <cstdint>
#include <random>
#include <vector>
#include "pool.h"

// Claims of 1..most lines from a pool of `cap` until `demand` lines were asked for.
template <class Counter>
static int check(unsigned cap, unsigned most, unsigned long long demand)
{
    std::mt19937 g(7);
    std::vector<std::uint8_t> owned(cap, 0);
    Counter cursor = 0;
    unsigned long long granted = 0;
    for (unsigned long long asked = 0; asked < demand;) {
        const unsigned used = 1u + g() % most;
        const Counter before = cursor;
        asked += used;
        cursor += used;
        const unsigned at = ade::claim_lines(before, cap, used);
        if (at == ade::kNoRoom) continue;
        if (at > cap || used > cap - at) return 1;
        for (unsigned k = 0; k < used; ++k) {
            if (owned[at + k]) return 1;
            owned[at + k] = 1;
        }
        granted += used;
    }
    return granted > cap ? 2 : 0;
}

int main()
{
    using Counter = unsigned long long;
    int bad = 0;
    bad |= check<Counter>(0u, 5u, 1ull << 12);
    bad |= check<Counter>(1000u, 40u, 1ull << 20);
    // demands that pass 2^32 many times, on a pool of 8 GB
    bad |= check<Counter>(1u << 26, 1u << 25, 60ull << 32);
    bad |= check<Counter>(1u << 26, 0x7fffffffu, 60ull << 32);
    if (check<std::uint32_t>(1u << 26, 1u << 25, 60ull << 32) == 0) bad |= 8;
    // a chunk's own count does not wrap either
    unsigned used = 6u;
    for (int r = 0; r < 169; ++r) {
        const unsigned next = ade::add_lines(used, 0x7fffffffu);
        if (next < used && used < 0x80000000u) bad |= 4;
        used = next;
    }
    if (used < 0x80000000u) bad |= 4;
    std::printf("%d\n", bad);
    return bad;
}
"""


def test_claims_never_overlap_beyond_2_to_32_lines(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "pool.cpp", tmp_path / "pool"
    src.write_text(SRC)
    inc = os.path.join(ROOT, "paper_2108_09488_gb300", "csrc")
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", inc, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout.strip() == "0"


def test_the_tables_counter_has_64_bits():
    src = open(os.path.join(ROOT, "paper_2108_09488_gb300", "csrc", "ade_internal.h")).read()
    assert "unsigned long long *cursor;" in src
