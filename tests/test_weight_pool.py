"""The counter of the weight table's pool of lines (csrc/pool.h), on the CPU: a sequence of claims
whose demands pass 2^32 lines several times over never gets a line twice and never lines beyond the
pool, whatever the interleaving of the compare-and-swaps."""
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

// Claims of 1..most lines from a pool of `cap` until `demand` lines were asked for; every third
// compare-and-swap first lets another claimant through.  plain_add: the counter that every demand is
// added to, which the check has to find out.
static int check(unsigned cap, unsigned most, unsigned long long demand, bool plain_add = false)
{
    std::mt19937 g(7);
    std::vector<std::uint8_t> owned(cap, 0);
    unsigned cursor = 0;
    unsigned long long asked = 0, granted = 0;
    int turn = 0;
    auto take = [&](unsigned at, unsigned used) {
        if (at == ade::kNoRoom) return true;
        if (at > cap || used > cap - at) return false;
        for (unsigned k = 0; k < used; ++k) {
            if (owned[at + k]) return false;
            owned[at + k] = 1;
        }
        granted += used;
        return true;
    };
    auto plain = [&](unsigned seen, unsigned next) {
        const unsigned was = cursor;
        if (was == seen) cursor = next;
        return was;
    };
    while (asked < demand) {
        const unsigned used = 1u + g() % most;
        asked += used;
        bool ok = true;
        auto crossed = [&](unsigned seen, unsigned next) {
            if (++turn % 3 == 0) {
                const unsigned other = 1u + g() % most;
                asked += other;
                ok = ok && take(ade::claim_lines(cursor, cap, other, plain), other);
            }
            return plain(seen, next);
        };
        unsigned at;
        if (plain_add) {
            at = cursor;
            cursor += used;
            if (!(at <= cap && cap - at >= used)) at = ade::kNoRoom;
            if (!take(at, used)) return 1;
            continue;
        }
        at = ade::claim_lines(cursor, cap, used, crossed);
        if (!ok || !take(at, used) || cursor > cap) return 1;
    }
    return granted > cap ? 2 : 0;
}

int main()
{
    int bad = 0;
    bad |= check(0u, 5u, 1ull << 12);
    bad |= check(1000u, 40u, 1ull << 20);
    // demands that pass 2^32 many times, on a pool of 8 GB
    bad |= check(1u << 26, 1u << 25, 60ull << 32);
    bad |= check(1u << 26, 0x7fffffffu, 60ull << 32);
    if (check(1u << 26, 1u << 25, 60ull << 32, true) == 0) bad |= 8;
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
