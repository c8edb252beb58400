"""A cooperative launch on a GPU with fewer free SMs than it reports, on a fake of the
CUDA runtime: the grid shrinks until it fits, other errors come back at once."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#pragma once
enum cudaError_t { cudaSuccess = 0, cudaErrorInvalidValue = 1, cudaErrorCooperativeLaunchTooLarge = 720 };
inline int g_last = 0;
inline cudaError_t cudaGetLastError() { cudaError_t e = (cudaError_t)g_last; g_last = 0; return e; }
"""

MAIN = r"""
#include "coop_launch.h"
int main() {
    int bad = 0;
    for (int fit = 1; fit <= 200; ++fit)
        for (int want = 1; want <= 152; ++want) {
            int ran = 0;
            const cudaError_t e = qsg::launch_resident_grid(want, [&](int n) {
                if (n > fit) return (cudaError_t)(g_last = cudaErrorCooperativeLaunchTooLarge);
                ran = n;
                return cudaSuccess;
            });
            const bool all = want <= fit;
            if (e != cudaSuccess || g_last != 0 || ran < 1 || ran > fit || (all && ran != want) || (!all && 2 * ran < fit)) ++bad;
        }
    int calls = 0;
    if (qsg::launch_resident_grid(152, [&](int) { ++calls; return cudaErrorInvalidValue; }) != cudaErrorInvalidValue || calls != 1) ++bad;
    calls = 0;  // not even one block fits: the error comes back
    if (qsg::launch_resident_grid(152, [&](int) { ++calls; return cudaErrorCooperativeLaunchTooLarge; }) == cudaSuccess || calls > 9) ++bad;
    return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_grid_shrinks_until_it_fits(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(FAKE)
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.run(["g++", "-std=c++17", "-I", str(tmp_path), "-I", os.path.join(ROOT, "paper_2310_07486_gb300", "csrc"),
                    str(tmp_path / "main.cpp"), "-o", exe], check=True, capture_output=True)
    assert subprocess.run([exe], timeout=60).returncode == 0
