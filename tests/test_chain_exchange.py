"""The exchanges between the layers of a dense chain: whatever the order of events, no reader misses the phase it waits for."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Every interleaving of a cluster of two CTAs and four layers, over all choices of which CTA owns columns of which layer.  A CTA is
# a reader (waits for the exchange behind layer l - 1, then the CTA's rows of layer l are on their way) and a writer (needs those
# rows where the CTA owns columns of layer l; then arrives at both CTAs' barriers, except behind the last layer).
PROGRAM = r"""
#include <cstdio>
#include <set>
#include <vector>
#include "exchange.h"

constexpr int kCtas = 2, kLayers = 4, kBarriers = ChainExchange::barriers(kLayers);
struct State {
    int reader[kCtas], writer[kCtas];      // layers done
    int arrived[kCtas][kBarriers];         // arrivals so far at each barrier of each CTA
    bool operator<(const State &o) const { return __builtin_memcmp(this, &o, sizeof(o)) < 0; }
};

// mbarrier.try_wait.parity: true where the phase in progress has the other parity, i.e. one of this parity was the last to complete
static bool seen(int arrivals, unsigned parity) { return ((unsigned)(arrivals / kCtas) & 1u) != (parity & 1u); }

static bool ends(int owns, long &states) {  // whether every interleaving ends
    std::set<State> known;
    std::vector<State> todo(1, State{});
    known.insert(todo[0]);
    while (!todo.empty()) {
        const State s = todo.back();
        todo.pop_back();
        ++states;
        bool moved = false, over = true;
        auto go = [&](const State &n) {
            moved = true;
            if (known.insert(n).second) todo.push_back(n);
        };
        for (int c = 0; c < kCtas; ++c) {
            over = over && s.reader[c] == kLayers && s.writer[c] == kLayers;
            const int r = s.reader[c], w = s.writer[c];
            if (r < kLayers && (r == 0 || seen(s.arrived[c][ChainExchange::barrier(r - 1)], ChainExchange::parity(r - 1)))) {
                State n = s;
                ++n.reader[c];
                go(n);
            }
            if (w < kLayers && (!((owns >> (c * kLayers + w)) & 1) || s.reader[c] > w)) {
                State n = s;
                ++n.writer[c];
                if (w + 1 < kLayers)
                    for (int o = 0; o < kCtas; ++o) ++n.arrived[o][ChainExchange::barrier(w)];
                go(n);
            }
        }
        if (!moved && !over) return false;
    }
    return true;
}

int main() {
    long states = 0;
    for (int owns = 0; owns < 1 << (kCtas * kLayers); ++owns)
        if (!ends(owns, states)) {
            printf("a reader waits for good: columns %#x\n", owns);
            return 1;
        }
    printf("ok %ld\n", states);
    return 0;
}
"""


def test_no_interleaving_leaves_a_reader_behind(tmp_path):
    src, exe = tmp_path / "exchange.cpp", tmp_path / "exchange"
    src.write_text(PROGRAM)
    csrc = os.path.join(ROOT, "paper_2509_16434_b200", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", csrc, "-o", str(exe), str(src)], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert run.returncode == 0 and run.stdout.startswith("ok"), run.stdout
