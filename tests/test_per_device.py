"""The launchers' per-device values (csrc/per_device.h): made once per device,
not kept when making fails, and the same for every thread that asks."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1409_0035_gb300", "csrc")

PROGRAM = r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"

static int fail(const char *what) { std::printf("%s\n", what); return 1; }

int main()
{
    static ccg::PerDevice<ccg::Residency> cache;
    std::atomic<int> made[2] = {{0}, {0}};
    std::atomic<int> wrong{0};
    auto ask = [&](int dev) {
        ccg::Residency r;
        const int rc = cache.get(dev, &r, [&](ccg::Residency &v) {
            made[dev] += 1;
            v.sms = 100 + dev;
            std::this_thread::yield();
            v.per_sm = 2 + dev;
            return 0;
        });
        if (rc != 0 || r.sms != 100 + dev || r.per_sm != 2 + dev) wrong += 1;
    };
    std::vector<std::thread> t;
    for (int i = 0; i < 16; ++i) t.emplace_back([&, i] { for (int j = 0; j < 200; ++j) ask((i + j) & 1); });
    for (auto &x : t) x.join();
    if (wrong) return fail("a thread saw another device's or a half made value");
    if (made[0] != 1 || made[1] != 1) return fail("made more than once");
    ccg::Residency r;
    int calls = 0;
    for (int i = 0; i < 2; ++i)
        if (cache.get(5, &r, [&](ccg::Residency &) { ++calls; return -6; }) != -6)
            return fail("status lost");
    if (calls != 2) return fail("a failure was kept");
    if (cache.get(1000, &r, [&](ccg::Residency &v) { v.sms = 7; return 0; }) != 0 || r.sms != 7)
        return fail("device beyond the table");
    return 0;
}
"""


def test_per_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "t"
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
