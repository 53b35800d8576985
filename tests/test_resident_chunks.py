"""Runs of sweeps as resident launches (no GPU; the launch is a fake): long runs go in
chunks, and a refused launch leaves its sweeps to the launches per colour."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <vector>
#include "mpr_resident.h"
using namespace mpr;
int main() {
    std::vector<int> runs;
    cudaError_t answer = cudaSuccess;
    size_t good = 100;  // launches that succeed before the answer
    const auto launch = [&](int m) {
        if (runs.size() >= good) return answer;
        runs.push_back(m);
        return cudaSuccess;
    };
    int done = -1;
    if (resident_chunks(0, launch, &done) != cudaSuccess || done != 0 || !runs.empty()) return 1;
    if (resident_chunks(7, launch, &done) != cudaSuccess || done != 7 || runs != std::vector<int>{7}) return 2;
    runs.clear();
    if (resident_chunks(2 * kMostSweeps + 5, launch, &done) != cudaSuccess || done != 2 * kMostSweeps + 5 ||
        runs != std::vector<int>{kMostSweeps, kMostSweeps, 5}) return 3;
    // fewer SMs than the device has: nothing launched, or the first chunk only
    for (cudaError_t refusal : {cudaErrorCooperativeLaunchTooLarge, cudaErrorNotSupported})
        for (good = 0; good < 2; ++good) {
            answer = refusal;
            runs.clear();
            if (resident_chunks(kMostSweeps + 1, launch, &done) != cudaSuccess ||
                done != (int)good * kMostSweeps) return 4;
        }
    // any other error is one
    good = 0;
    answer = cudaErrorInvalidValue;
    if (resident_chunks(3, launch, &done) != cudaErrorInvalidValue || done != 0) return 5;
    return 0;
}
"""


def test_long_runs_and_refused_launches(tmp_path):
    cxx = shutil.which("g++")
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if cxx is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or no CUDA headers")
    src, exe = tmp_path / "chunks.cc", tmp_path / "chunks"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_1710_03038_gb300", "csrc"),
                    "-I", os.path.join(ROOT, "include"), "-I", cuda, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
