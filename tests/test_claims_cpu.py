"""Claims of a server's trials, on host threads (no GPU needed): the claim word's
functions are the device's own.  Claimers look at a record, and the record may be
used up, freed and taken by a later failure before they claim."""
import os
import shutil
import subprocess

import pytest

from paper_2507_00254_gb300 import build as libbuild

PROGRAM = r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "bpsf_internal.h"
using namespace bpsf;
typedef unsigned long long u64;

static std::atomic<u64> cell;
static auto swap_cell = [](u64 old, u64 next) { cell.compare_exchange_strong(old, next); return old; };

// A claim that comes late takes nothing and leaves the record's word alone.
static int late(int T, int want) {
    int bad = 0, first = -1;
    for (u64 q : {0ull, 5ull, (1ull << 31) + 7, (1ull << 50) - 1})
        for (u64 later : {q + 1, q + 32, q + (1ull << 32)})
            for (int seen = 0; seen < T; seen += T / 4 + 1)
                for (int taken : {0, seen, T}) {
                    cell = claim_word(later, taken);
                    bad += claim_trials(claim_word(q, seen), q, want, T, &first, swap_cell) != 0;
                    bad += cell != claim_word(later, taken);
                    bad += claim_taken(cell, q, T) != T || claim_taken(cell, later, T) != taken;
                    // In time: what is left, from the first one on.
                    cell = claim_word(q, seen);
                    const int n = claim_trials(cell, q, want, T, &first, swap_cell);
                    bad += n != (T - seen < want ? T - seen : want) || first != seen || cell != claim_word(q, seen + n);
                }
    return bad;
}

// Threads claim from one record that holds failure after failure: every trial of
// every failure is taken once.
static int race(int threads, int failures, int T) {
    std::vector<std::vector<std::atomic<int>>> got(failures);
    for (auto &v : got) v = std::vector<std::atomic<int>>(T);
    std::vector<std::atomic<int>> done(failures);
    std::atomic<u64> published{0};
    cell = claim_word(0, 0);
    auto work = [&](int t) {
        unsigned x = 12345u + t;
        for (;;) {
            const u64 q = published.load();
            if (q >= (u64)failures) return;
            const u64 word = cell.load();
            x = x * 1664525u + 1013904223u;
            if ((x >> 28) == 0) std::this_thread::yield();  // late
            int first = 0;
            const int n = claim_trials(word, q, 1 + (int)((x >> 16) % 9u), T, &first, swap_cell);
            for (int k = 0; k < n; ++k) ++got[q][first + k];
            if (n && (done[q] += n) == T) {  // the last trial: the record's next failure
                cell = claim_word(q + 1, 0);
                published = q + 1;
            }
        }
    };
    std::vector<std::thread> ts;
    for (int t = 0; t < threads; ++t) ts.emplace_back(work, t);
    for (auto &t : ts) t.join();
    int bad = 0;
    for (auto &v : got)
        for (auto &n : v) bad += n != 1;
    return bad;
}

int main() {
    const int a = late(63, 32) + late(4096, 32) + late(1, 1), b = race(8, 3000, 63);
    printf("%d %d\n", a, b);
    return a || b;
}
"""


def test_late_and_contended_claims(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "claims.cpp", tmp_path / "claims"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O2", "-pthread", "-D__host__=", "-D__device__=", "-I", libbuild.CSRC,
                    str(src), "-o", str(exe)], check=True, cwd=os.path.dirname(libbuild.CSRC))
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
