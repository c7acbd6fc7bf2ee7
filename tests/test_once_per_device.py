"""Kernel attributes are set once per device, not once per process: the host
class that sees to it runs its function for every device, again after a
failure, and no second time after a success; and no launcher keeps such a
setting in a process-wide flag."""
from __future__ import annotations

import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2402_00665_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "once_per_device.cuh"
int main() {
    lbvh::OncePerDevice once;
    std::vector<int> ran(80, 0);
    auto go = [&](int dev, bool result) { return once(dev, [&] { ++ran[dev]; return result; }); };
    for (int dev : {0, 1, 63, 64, 79}) {
        if (go(dev, false) || ran[dev] != 1) return 1;  // a failure is reported and not remembered
        if (!go(dev, true) || ran[dev] != 2) return 2;
        if (!go(dev, true)) return 3;
        if (ran[dev] != (dev < 64 ? 2 : 3)) return 4;   // a success is, for the devices it has room for
    }
    if (!go(2, true) || ran[2] != 1) return 5;          // another device still runs it
    lbvh::OncePerDevice other;
    std::atomic<int> calls{0}, bad{0};
    std::vector<std::thread> threads;
    for (int t = 0; t < 8; ++t)
        threads.emplace_back([&] {
            for (int k = 0; k < 1000; ++k)
                if (!other(k % 4, [&] { ++calls; return true; }) || calls == 0) ++bad;
        });
    for (auto &t : threads) t.join();
    if (bad || calls < 4 || calls > 32) return 6;
    std::puts("ok");
    return 0;
}
"""


def test_runs_once_for_every_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("needs a C++ compiler")
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.returncode


def test_every_kernel_attribute_is_set_per_device():
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        text = open(path).read()
        if "cudaFuncSetAttribute(" in text:
            assert "OncePerDevice" in text, path
        assert not re.search(r"static const \w+ \w+ = \[\][^;]*cudaFuncSetAttribute", text), path
