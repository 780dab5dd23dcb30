"""How the halo convolutions divide an SM's shared memory, as the library's own planner does it, and how the ring in it is handed over."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Forward passes (Ci -> Co) and input gradients (Co -> Ci) on grids of w x h: the slots a CTA has against those that fit beside what the
# kernel needs, counted here: weights, staging, two alignments, 25 barriers, two words and three vectors of 256 floats.
PROGRAM = r"""
#include <cstdio>
#include "halo_plan.h"
using namespace halo;

int main() {
    const int layers[][3] = {{16, 32, 0}, {16, 48, 0}, {32, 32, 0}, {32, 48, 0}, {32, 64, 0}, {64, 64, 0}, {16, 32, 1}, {16, 48, 1},
                             {16, 64, 1}, {32, 32, 1}, {32, 48, 1}, {32, 64, 1}, {32, 128, 1}, {64, 96, 1}};
    long plans = 0, fewer = 0;
    for (const auto &l : layers)
        for (int w = 2; w <= 120; ++w)
            for (int h = w * 3 / 4; h <= w; ++h) {
                const int Ci = l[0], Co = l[1], from = l[2] ? Co : Ci;
                Args a = {};
                a.CB = from % 64 == 0 ? 64 : (from % 32 == 0 ? 32 : 16);
                a.rb = 2 * a.CB;
                a.nchunks = from / a.CB;
                a.nplanes = l[2] ? 1 : 4;
                a.nloads = l[2] ? a.nchunks : 4;
                a.N = l[2] ? 4 * Ci : Co;
                a.w_chunk = 9u * (l[2] ? Ci : Co) * a.rb;
                if (h < 2 || !plan(a, w, h, 512)) continue;
                ++plans;
                const size_t room = a.per_sm == 2 ? kSmemMax / 2 - 512 : kSmemMax, weights = ((size_t)a.nchunks * a.w_chunk + 1023) & ~size_t(1023);
                const size_t need = weights + (size_t)(a.nbuf * a.neg) * a.stg_bytes + 2 * 1024 + 25 * 8 + 2 * 4 + 3 * 256 * 4;
                const int fit = (int)((room - need) / a.slot_bytes);
                if (a.slots < (fit < kMaxSlots ? fit : kMaxSlots) && ++fewer <= 5)
                    printf("%d -> %d %s %d x %d: %d slots, %d fit\n", Ci, Co, l[2] ? "input gradient" : "forward", w, h, a.slots, fit);
            }
    printf("%ld plans, %ld with fewer slots than fit\n", plans, fewer);
    return plans < 1000 || fewer != 0;
}
"""


def _compile(src, exe, *more):
    csrc = os.path.join(ROOT, "paper_2509_16434_b200", "csrc")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O2", *more, "-I", csrc, "-I", os.path.join(cuda, "include"), "-o", str(exe), str(src)], check=True)


def test_the_ring_takes_no_room_from_kernels_without_one(tmp_path):
    src, exe = tmp_path / "room.cpp", tmp_path / "room"
    src.write_text(PROGRAM)
    _compile(src, exe)
    run = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stdout



# Every interleaving of the ring's hand-overs for runs that cross ends of images, on planned grids: two epilogue groups on alternate
# tiles, builders of both sets, and the sums.  A wait that a barrier's parity lets pass before its time, or one that never passes
# although nothing else can move, is an error.  FAULT plants one: 1, each set's first builder gives back the row groups that end in the
# stages of its own set; 2, a builder waits for the pixels of its own trip only.
RING = r"""
#include <cstdio>
#include <cstdlib>
#include <unordered_set>
#include <vector>
#include "halo_plan.h"
using namespace halo;

static bool gives_back(int builder, int s, int end) {
    if (FAULT == 1) return (builder & 3) == 0 && end > ring_summed(s) - kStagePx;
    return ring_gives_back(builder);
}

static int needs(int builder, int s, int total) {
    const int end = s * kStagePx + ((builder & 3) + 1) * kTrip;
    if (FAULT == 2) return end < total ? end : total;
    return ring_needs(s, total);
}

struct Run {
    int groups, xsegs;        // barriers, tiles of a row group
    std::vector<int> end;     // of row group n, in pixels of the run
    int total, nstages, ntiles;
    std::vector<int> builder; // the builders that are followed; a set hands a stage over when all of its builders among them have
};

constexpr int kMost = 4;
struct State {
    uint64_t given;                            // row groups given back
    uint8_t tile[2], writing[2];               // next tile of each epilogue group (of both's); whether it has been let in
    uint8_t stage[kMost], step[kMost];         // builders: next stage; 0 not let in, 1 let in, 2 has given back
    uint8_t walked[kMost], seen[kMost];        // row groups gone through to be given back; seen in the ring
    uint8_t sums, pad[3];                      // stages summed
};
static_assert(sizeof(State) == 32, "");
struct Hash {
    size_t operator()(const State &s) const {
        uint64_t h = 1469598103934665603ull, w[4];
        __builtin_memcpy(w, &s, 32);
        for (uint64_t x : w) h = (h ^ x) * 1099511628211ull, h ^= h >> 29;
        return h;
    }
};
struct Same { bool operator()(const State &a, const State &b) const { return __builtin_memcmp(&a, &b, sizeof a) == 0; } };

// mbarrier.try_wait.parity after `complete` phases
static bool passes(int complete, int parity) { return (complete & 1) != (parity & 1); }

static const char *follow(const Run &r, long &states) {
    std::unordered_set<State, Hash, Same> known;
    State first = {};
    const int nb = (int)r.builder.size(), G = r.groups, ngroups = (int)r.end.size();
    first.tile[1] = 1;
    for (int b = 0; b < nb; ++b) first.stage[b] = (uint8_t)(r.builder[b] >> 2);
    std::vector<State> todo(1, first);
    known.insert(first);
    while (!todo.empty()) {
        const State s = todo.back();
        todo.pop_back();
        ++states;
        bool moved = false;
        auto go = [&](const State &n) {
            moved = true;
            if (known.insert(n).second) todo.push_back(n);
        };
        auto tiles_done = [&](int g) {  // of row group g
            int n = 0;
            for (int t = g * r.xsegs; t < (g + 1) * r.xsegs; ++t) n += t < s.tile[t & 1];
            return n;
        };
        auto given = [&](int i) {  // phases of gempty[i]
            int n = 0;
            for (int g = i; g < ngroups; g += G) n += (int)(s.given >> g & 1);
            return n;
        };
        auto full = [&](int i) {  // phases of gfull[i]
            int n = 0;
            for (int g = i; g < ngroups; g += G) n += tiles_done(g);
            return n / r.xsegs;
        };
        auto handed = [&](int k) {  // whether stage k has been handed over
            for (int b = 0; b < nb; ++b)
                if ((r.builder[b] >> 2) == (k & 1) && s.stage[b] <= k) return false;
            return true;
        };
        for (int e = 0; e < 2; ++e) {
            const int t = s.tile[e], g = t / r.xsegs;
            if (t >= r.ntiles) continue;
            State n = s;
            if (s.writing[e]) {
                n.writing[e] = 0;
                n.tile[e] += 2;
                go(n);
            } else if (passes(given(g % G), (g / G & 1) ^ 1)) {
                if (g >= G && !(s.given >> (g - G) & 1)) return "an epilogue group writes over pixels that have not been given back";
                n.writing[e] = 1;
                go(n);
            }
        }
        for (int b = 0; b < nb; ++b) {
            const int k = s.stage[b], w = s.walked[b];
            if (k >= r.nstages) continue;
            State n = s;
            if (s.step[b] == 0) {  // stage k - kWinStages has been summed
                if (k >= kWinStages && s.sums <= k - kWinStages) continue;
                n.step[b] = 1;
                go(n);
            } else if (s.step[b] == 1) {
                if (w < ngroups && r.end[w] <= ring_summed(k)) {
                    if (gives_back(r.builder[b], k, r.end[w])) {
                        if (r.end[w] > s.sums * kStagePx) return "pixels are given back that have not been summed";
                        n.given |= 1ull << w;
                    }
                    ++n.walked[b];
                } else n.step[b] = 2;
                go(n);
            } else {
                const int g = s.seen[b];
                if (g == 0 || r.end[g - 1] < needs(r.builder[b], k, r.total)) {
                    if (!passes(full(g % G), g / G & 1)) continue;
                    if (tiles_done(g) < r.xsegs) return "a builder takes pixels for written that are not";
                    ++n.seen[b];
                } else {
                    n.step[b] = 0;
                    n.stage[b] += 2;
                }
                go(n);
            }
        }
        if (s.sums < r.nstages && handed(s.sums) && (s.sums + 1 == r.nstages || handed(s.sums + 1))) {
            State n = s;
            ++n.sums;
            go(n);
        }
        if (!moved && s.sums < r.nstages) return "nothing can move";
    }
    return nullptr;
}

// Frame rows and columns, output channels of the second layer, row groups of the run's first image, its pixels in front of the run,
// stages; then the builders to follow.
int main(int argc, char **argv) {
    std::vector<int> v;
    for (int i = 1; i < argc; ++i) v.push_back(atoi(argv[i]));
    Run r;
    r.builder.assign(v.begin() + 6, v.end());
    const int Hi = (v[0] + 1) / 2, Wi = v[1] / 2, Co = v[2];
    Args a = {};
    First f = {};
    a.CB = Co % 64 == 0 ? 64 : (Co % 32 == 0 ? 32 : 16);
    a.rb = 2 * a.CB;
    a.nloads = a.nchunks = Co / a.CB;
    a.N = 128;
    a.w_chunk = 9u * 32 * a.rb;
    if (!plan_first(a, f, Hi, Wi, 512)) return printf("no plan\n"), 2;
    r.groups = f.groups;
    r.xsegs = a.xsegs;
    r.nstages = v[5];
    r.total = r.nstages * kStagePx - 40;
    int k = a.ysegs - v[3] % a.ysegs;
    for (int end = -v[4]; r.end.empty() || r.end.back() < r.total; k = (k + 1) % a.ysegs)
        r.end.push_back(end += k % a.ysegs == a.ysegs - 1 ? f.last_px : f.group_px);
    r.ntiles = (int)r.end.size() * r.xsegs;
    if (r.end[0] <= 0 || r.end.size() > 60 || r.ntiles > 250 || r.builder.size() > kMost) return 2;
    long states = 0;
    const char *wrong = follow(r, states);
    printf("%d row groups, %d in flight, of %d px, the last of an image %d, %d tiles each: %s (%ld states)\n", (int)r.end.size(), r.groups,
           f.group_px, f.last_px, r.xsegs, wrong ? wrong : "ok", states);
    return wrong != nullptr;
}
"""

# frames, channels, row groups of the run's first image, pixels in front of the run: odd and even numbers of row groups in flight, short
# last ones, several tiles each, runs that start in and at row groups
RUNS = [(124, 164, 64, 2, 16), (180, 240, 64, 2, 80), (69, 90, 64, 1, 16), (162, 108, 64, 2, 112), (205, 126, 64, 1, 16), (84, 112, 64, 1, 64),
        (110, 146, 64, 3, 8), (240, 320, 64, 2, 0), (201, 268, 32, 2, 100), (120, 160, 64, 1, 0)]


def _ring(tmp_path, fault, builders):
    """The verdicts on all runs, in order."""
    src, exe = tmp_path / "ring.cpp", tmp_path / "ring"
    src.write_text(RING)
    _compile(src, exe, f"-DFAULT={fault}")
    found = []
    for r in RUNS:
        run = subprocess.run([str(exe)] + [str(v) for v in r + (30,) + builders], capture_output=True, text=True, timeout=300)
        assert run.returncode in (0, 1), run.stdout
        found.append(run.stdout)
    return found


@pytest.mark.parametrize("builders", [(0, 4), (0, 4, 1), (0, 4, 2, 5)])
def test_the_ring_is_handed_over_in_order(tmp_path, builders):
    assert all(": ok" in o for o in _ring(tmp_path, 0, builders))


def test_two_that_give_back_are_found_out(tmp_path):
    """Released by two builders, a row group can be given back before the one in front of it: seen where their number is odd."""
    assert all("not been given back" in o for o in _ring(tmp_path, 1, (0, 4))[:3])


def test_a_builder_that_falls_behind_is_found_out(tmp_path):
    """Builder 1, waiting for its own trip's pixels alone, misses a row group of 54 pixels that is filled twice meanwhile."""
    assert "nothing can move" in _ring(tmp_path, 2, (0, 4, 1))[3]
