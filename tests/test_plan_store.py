"""The store of prepared launches: what is asked for in every call stays, whatever else comes in and goes."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <new>
#include "plan_store.h"

static bool no_memory = false;
void *operator new(size_t n) {
    if (no_memory) throw std::bad_alloc();
    return malloc(n);
}
void operator delete(void *p) noexcept { free(p); }
void operator delete(void *p, size_t) noexcept { free(p); }

struct Key { long long op; const void *p; };
#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)

int main() {
    PlanStore<Key, long long> s(64);
    const Key every[3] = {{1, nullptr}, {2, nullptr}, {3, nullptr}};
    int misses = 0;
    for (long long call = 0; call < 1000; ++call) {  // a call: three operations at fixed addresses, one at a new one
        for (const Key &k : every) {
            const long long *v = s.find(k);
            if (v) CHECK(*v == 10 * k.op);
            else { ++misses; s.put(k, 10 * k.op); }
        }
        const Key passing{4, (const void *)(1000 + call)};
        CHECK(!s.find(passing));
        s.put(passing, 1000 + call);
        CHECK(s.find(passing) && *s.find(passing) == 1000 + call);
        CHECK(s.size() <= 64);
    }
    CHECK(misses == 3);  // prepared once each
    CHECK(s.size() == 64);
    CHECK(!s.find(Key{4, (const void *)(1000 + 900)}));  // long gone
    CHECK(s.find(Key{4, (const void *)(1000 + 990)}));
    no_memory = true;
    s.put(Key{5, nullptr}, 5);  // returns
    CHECK(!s.find(Key{5, nullptr}) && s.find(every[0]));
    no_memory = false;
    s.put(Key{5, nullptr}, 5);
    CHECK(s.find(Key{5, nullptr}) && *s.find(Key{5, nullptr}) == 5 && s.size() <= 64);
    s.clear();
    CHECK(s.size() == 0 && !s.find(every[0]));
    puts("ok");
    return 0;
}
"""


def test_operations_of_every_call_outlive_passing_ones(tmp_path):
    src, exe = tmp_path / "store.cpp", tmp_path / "store"
    src.write_text(PROGRAM)
    csrc = os.path.join(ROOT, "paper_2509_16434_b200", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", csrc, "-o", str(exe), str(src)], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert run.returncode == 0 and run.stdout.strip() == "ok", run.stdout


REPLAY = r"""
#include <cstdio>
#include "launch.cuh"

// stands in for the runtime's launch: remembers the arguments' values
static int calls, first[4];
static double second[4];
extern "C" cudaError_t CUDARTAPI cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *, void **argv) {
    memcpy(&first[calls], argv[0], sizeof(int));
    memcpy(&second[calls], argv[1], sizeof(double));
    ++calls;
    return cudaSuccess;
}
void ppo_count_launches(int) {}
#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)

int main() {
    Recording made;
    ppo_recording = &made;
    int a = 7;
    double end = 1.5;
    void *argv[] = {&a, &end};
    const size_t sizes[] = {sizeof(a), sizeof(end)};
    ppo_record((const void *)main, dim3(1), dim3(1), 0, false, argv, sizes, 2);
    ppo_recording = nullptr;
    const double other = 2.5;
    CHECK(ppo_replay(made.launches, nullptr) == PPO_OK && calls == 1 && first[0] == 7 && second[0] == 1.5);
    CHECK(ppo_replay(made.launches, nullptr, &other, sizeof(other)) == PPO_OK && calls == 2 && first[1] == 7 && second[1] == 2.5);
    CHECK(ppo_replay(made.launches, nullptr) == PPO_OK && calls == 3 && second[2] == 1.5);  // the record keeps its own
    CHECK(ppo_replay(made.launches, nullptr, &other, sizeof(float)) == PPO_ERR_CUDA && calls == 3);  // another argument
    puts("ok");
    return 0;
}
"""


def test_a_replay_may_have_another_last_argument(tmp_path):
    src, exe = tmp_path / "replay.cu", tmp_path / "replay"
    src.write_text(REPLAY)
    from paper_2509_16434_b200 import build
    csrc = os.path.join(ROOT, "paper_2509_16434_b200", "csrc")
    subprocess.run([build.NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-cudart", "shared", "-I", csrc, "-o", str(exe),
                    str(src), os.path.join(csrc, "launch.cu")], check=True)
    lib = os.path.join(os.path.dirname(os.path.dirname(build.NVCC)), "lib64")
    run = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60, env=dict(os.environ, LD_LIBRARY_PATH=lib))
    assert run.returncode == 0 and run.stdout.strip() == "ok", run.stdout + run.stderr
