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
