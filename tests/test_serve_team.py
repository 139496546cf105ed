"""The protocol by which CTAs agree on a served query's team (csrc/serve_team.h),
run by host threads: whatever the order in which the leader and the members run,
and whoever's wait runs out first, all of them get the same size, and their
ranks are the numbers below it."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <atomic>
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <thread>
#include <vector>
#include "serve_team.h"
using namespace abfs;

static unsigned long long clock_ns() {
    return std::chrono::duration_cast<std::chrono::nanoseconds>(
               std::chrono::steady_clock::now().time_since_epoch()).count();
}
struct Io {
    std::atomic<unsigned long long>* word;
    unsigned long long load() { return word->load(); }
    unsigned long long close() { return word->fetch_and(~kJoinOpen); }
    unsigned long long now() { return clock_ns(); }
};
static void nap(std::mt19937& r, unsigned us) {
    if (r() % 2) std::this_thread::sleep_for(std::chrono::microseconds(r() % us));
}

int main() {
    std::atomic<unsigned long long> word{0};
    unsigned given_up = 0;
    for (unsigned round = 0; round < 400; ++round) {
        std::mt19937 rng(round);
        const uint32_t wanted = 2 + rng() % 5, ctas = 1 + rng() % 6;
        word = join_opened(word, wanted);
        std::atomic<int> go{0};
        std::vector<uint32_t> size(ctas + 1, 0), rank(ctas + 1, ~0u);
        std::vector<std::thread> th;
        // the leader comes late in half of the rounds, after the members' waits
        th.emplace_back([&] {
            std::mt19937 r(round * 31 + 7);
            while (!go) {}
            if (round % 2) std::this_thread::sleep_for(std::chrono::microseconds(600));
            Io io{&word};
            rank[0] = 0;
            size[0] = team_form(io, true, 100000, round % 3 ? 0 : 400000);
        });
        for (uint32_t c = 1; c <= ctas; ++c)
            th.emplace_back([&, c] {
                std::mt19937 r(round * 31 + 7 + c);
                while (!go) {}
                nap(r, 300);
                unsigned long long w = word;
                while (join_room(w)) {
                    if (!word.compare_exchange_strong(w, w + 1)) continue;
                    rank[c] = join_count(w);
                    nap(r, 200);
                    Io io{&word};
                    size[c] = team_form(io, false, 150000);
                    break;
                }
            });
        go = 1;
        for (auto& t : th) t.join();
        std::vector<int> seen(wanted, 0);
        uint32_t joined = 0;
        for (uint32_t c = 0; c <= ctas; ++c) {
            if (rank[c] == ~0u) continue;
            ++joined;
            if (size[c] != size[0] || rank[c] >= size[c] || seen[rank[c]]++) {
                std::printf("round %u: cta %u has rank %u of %u, the leader's team is %u\n", round, c,
                            rank[c], size[c], size[0]);
                return 1;
            }
        }
        if (joined != size[0]) return 2;
        given_up += size[0] < wanted;
    }
    std::printf("%u\n", given_up);
    return given_up ? 0 : 3;
}
"""


def test_everybody_gets_the_same_team(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "team.cpp", tmp_path / "team"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-I",
                    os.path.join(ROOT, "paper_1906_03113_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
