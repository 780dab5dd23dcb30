"""What is set up once per device may be asked for by several threads at once."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"

#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)

int main() {
    static PerDevice<int> numbers;
    std::atomic<int> made{0}, wrong{0};
    std::vector<std::thread> all;
    for (int t = 0; t < 4; ++t)
        all.emplace_back([&] {
            for (int i = 0; i < 2000; ++i)
                if (numbers.get(i % 64, [&] { ++made; return i % 64 + 100; }) != i % 64 + 100) ++wrong;
        });
    for (auto &t : all) t.join();
    CHECK(wrong == 0 && made >= 64 && made <= 4 * 64);
    static PerDevice<bool> done;
    CHECK(!done.get(3, [] { return false; }) && done.get(3, [] { return true; }) && done.get(3, [] { return false; }));
    CHECK(!done.get(-1, [] { return true; }) && !done.get(64, [] { return true; }));
    puts("ok");
    return 0;
}
"""


def test_threads_that_ask_at_once_do_not_race(tmp_path):
    src, exe = tmp_path / "per_device.cpp", tmp_path / "per_device"
    src.write_text(PROGRAM)
    csrc = os.path.join(ROOT, "paper_2509_16434_b200", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=thread", "-I", csrc, "-o", str(exe), str(src)], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert run.returncode == 0 and run.stdout.strip() == "ok", run.stdout + run.stderr[-2000:]


def test_every_table_by_device_is_one_of_these():
    csrc = os.path.join(ROOT, "paper_2509_16434_b200", "csrc")
    for name in sorted(os.listdir(csrc)):
        text = open(os.path.join(csrc, name)).read()
        assert not re.search(r"static [\w ]+\*?\w+(\[\d+\])?\[64\]", text), name
