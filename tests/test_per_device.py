"""The launchers' per-device numbers (csrc/per_device.h) under concurrent first
calls: a program with eight threads, built with the thread sanitizer, in which a
thread that finds a device ready must see both numbers and what was set up
before they were published."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1606_06117_gb300", "csrc")

PROGRAM = """
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
static sl::ResidencyCache cache;
static int opted_in[64];          // set up before a device is published
int main()
{
    std::atomic<int> bad{0};
    std::vector<std::thread> t;
    for (int k = 0; k < 8; ++k)
        t.emplace_back([&, k] {
            for (int i = 0; i < 4000; ++i) {
                const int dev = i % 64;
                sl::Residency r;
                if (cache.get(dev, r)) {
                    if (r.sms != 100 + dev || r.per_sm != 1 + dev % 4 || opted_in[dev] != 1) ++bad;
                } else if (dev % 8 == k) {   // one thread sets a device up here
                    opted_in[dev] = 1;
                    cache.set(dev, {100 + dev, 1 + dev % 4});
                }
            }
        });
    for (auto &x : t) x.join();
    std::printf("bad %d\\n", bad.load());
    return bad.load() != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_both_numbers_are_published_together(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    build = subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=thread", "-pthread", "-I", CSRC, str(src), "-o", str(exe)],
                           capture_output=True, text=True)
    if build.returncode != 0 and "tsan" in build.stderr:
        pytest.skip("no thread sanitizer")
    assert build.returncode == 0, build.stderr
    run = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    if "unexpected memory mapping" in run.stderr:
        pytest.skip("the thread sanitizer does not start under this kernel's address layout")
    assert run.returncode == 0 and "data race" not in run.stderr, run.stdout + run.stderr[:2000]
    assert run.stdout == "bad 0\n"
