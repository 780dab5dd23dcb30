"""How the halo convolutions divide an SM's shared memory, as the library's own planner does it, compiled on its own."""
import os
import subprocess

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


def _run(tmp_path, text, name):
    src, exe = tmp_path / (name + ".cpp"), tmp_path / name
    src.write_text(text)
    csrc = os.path.join(ROOT, "paper_2509_16434_b200", "csrc")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", csrc, "-I", os.path.join(cuda, "include"), "-o", str(exe), str(src)], check=True)
    return subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)


def test_the_ring_takes_no_room_from_kernels_without_one(tmp_path):
    run = _run(tmp_path, PROGRAM, "room")
    assert run.returncode == 0, run.stdout
