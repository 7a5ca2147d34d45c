"""The per-device values of the launchers (csrc/device_cache.h), on the CPU with made-up devices: a
value belongs to its device, is formed once however many threads ask for it first, is complete for
each of them, and an error is passed on and tried again."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2410_11625_gb300", "csrc")

PROGRAM = r"""
#include "device_cache.h"
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>

struct Value { int a = 0, b = 0; };

int main()
{
    static PerDevice<Value> known;
    std::atomic<int> fills[3] = {}, wrong{0}, go{0};
    std::vector<std::thread> threads;
    for (int t = 0; t < 12; ++t)
        threads.emplace_back([&, t] {
            const int dev = t % 3;
            while (!go.load()) {}
            for (int k = 0; k < 100; ++k) {
                Value v;
                const int e = known.get(dev, [&](Value &w) {
                    fills[dev]++;
                    w.a = 100 + dev;
                    std::this_thread::sleep_for(std::chrono::milliseconds(5));  // half filled
                    w.b = 200 + dev;
                    return 0;
                }, v);
                wrong += e != 0 || v.a != 100 + dev || v.b != 200 + dev;
            }
        });
    go = 1;
    for (auto &t : threads) t.join();
    if (wrong || fills[0] != 1 || fills[1] != 1 || fills[2] != 1) return 1;

    static PerDevice<Value> other;
    Value v;
    int calls = 0;
    auto fail_once = [&](Value &w) { w.a = 7; return ++calls == 1 ? 5 : 0; };
    if (other.get(4, fail_once, v) != 5 || other.get(4, fail_once, v) != 0 || v.a != 7 || calls != 2) return 2;
    if (other.get(4, fail_once, v) != 0 || calls != 2) return 3;
    // a device beyond the table is asked every time
    if (other.get(1000, fail_once, v) != 0 || other.get(-1, fail_once, v) != 0 || calls != 4) return 4;
    std::puts("ok");
    return 0;
}
"""


def test_one_value_per_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "cache.cpp", tmp_path / "cache"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.returncode


def test_launchers_keep_no_unkeyed_values():
    """A value in a plain static belongs to whichever device was current first, and is written
    without a lock by every thread that comes early."""
    import re
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for line in re.findall(r"^ +static (?!constexpr|_assert|cudaError_t |size_t smem|std::atomic|std::mutex|PerDevice)[^\n(]*;", text, flags=re.M):
            assert re.search(r"\[64\]", line), (name, line.strip())  # by device, under a lock
