"""CPU: values made once per device and read from any thread (csrc/gabp_per_device.h), under the
compiler's thread sanitizer."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_12968_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "gabp_per_device.h"
struct Limits { int a = 0, b = 0; };
static gabp::PerDevice<Limits> cache;
static int made[70], failed[70];   // written under the cache's lock only (devices 0 .. 63)
int main() {
    std::vector<std::thread> ts;
    std::atomic<int> bad{0};
    for (int t = 0; t < 8; ++t)
        ts.emplace_back([&, t] {
            for (int r = 0; r < 2000; ++r) {
                const int dev = (t + r) % 4 == 3 ? 63 : (t + r) % 4;
                Limits l;
                const int e = cache.get(dev, l, [&](Limits &v) {
                    if (failed[dev]++ < 2) return 7;   // the first two attempts fail: not kept
                    ++made[dev];
                    v.a = 100 + dev;
                    v.b = 200 + dev;
                    return 0;
                });
                if (e == 0 ? l.a != 100 + dev || l.b != 200 + dev : e != 7) ++bad;
            }
        });
    for (auto &t : ts) t.join();
    Limits l;
    for (int dev : {-1, 64})   // outside the table: made on every call
        for (int r = 0; r < 2; ++r)
            if (cache.get(dev, l, [&](Limits &v) { v.a = ++made[69]; return 0; }) || l.a != made[69]) ++bad;
    for (int dev : {0, 1, 2, 63})
        if (made[dev] != 1 || failed[dev] != 3) ++bad;
    std::printf("%d\n", bad.load() + (made[69] != 4));
    return bad.load() || made[69] != 4;
}
"""


def test_per_device_values_from_several_threads(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", str(tmp_path / "t")
    src.write_text(PROGRAM)
    r = subprocess.run([cxx, "-std=c++17", "-O2", "-fsanitize=thread", "-pthread", "-I", CSRC, str(src), "-o", exe],
                       capture_output=True, text=True)
    if r.returncode and "tsan" in r.stderr:
        pytest.skip("no thread sanitizer")
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    if "unexpected memory mapping" in r.stderr:
        pytest.skip("the thread sanitizer does not run on this kernel")
    assert r.returncode == 0 and r.stdout.strip() == "0", r.stdout + r.stderr
