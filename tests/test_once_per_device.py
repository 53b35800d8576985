"""The per-device settings of the kernels (no GPU): made once on every device, again after
a failure, from any thread."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "mpr_once.h"
int main() {
    mpr::OncePerDevice once;
    int calls = 0;
    const auto set = [&](int status) { return [&calls, status] { ++calls; return status; }; };
    if (once(0, set(7)) != 7 || calls != 1) return 1;   // a failure is not remembered
    if (once(0, set(0)) != 0 || calls != 2) return 2;
    if (once(0, set(7)) != 0 || calls != 2) return 3;   // made on device 0
    if (once(1, set(0)) != 0 || calls != 3) return 4;   // another device has its own
    if (once(1, set(7)) != 0 || once(0, set(7)) != 0 || calls != 3) return 5;
    if (once(64, set(0)) != 0 || once(64, set(0)) != 0 || calls != 5) return 6;
    mpr::OncePerDevice shared;
    std::vector<std::thread> ts;
    for (int t = 0; t < 8; ++t)
        ts.emplace_back([&shared, t] { for (int k = 0; k < 1000; ++k) shared((k + t) % 60, [] { return 0; }); });
    for (auto& t : ts) t.join();
    for (int d = 0; d < 60; ++d)
        if (shared(d, [] { return 7; }) != 0) return 7;
    return 0;
}
"""


def test_a_setting_is_made_once_on_every_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "once.cc", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "paper_1710_03038_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
