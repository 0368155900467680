"""The shared-memory opt-in (csrc/smem_optin.h) compiled by the host compiler against a counting
stand-in of the CUDA runtime: once per kernel and device, again on another device, not
remembered when it failed, and correct from several threads."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1104_5497_gb300", "csrc")

RUNTIME = """
#pragma once
#include <atomic>
typedef int cudaError_t;
enum { cudaSuccess = 0, cudaFuncAttributeMaxDynamicSharedMemorySize = 8 };
extern thread_local int now;              // the current device
extern std::atomic<int> sets[3][70];      // attribute calls by kernel (its number) and device
extern std::atomic<int> fails;            // calls that are still to fail
inline cudaError_t cudaGetDevice(int *d) { *d = now; return 0; }
template <class F> cudaError_t cudaFuncSetAttribute(F *f, int attr, int bytes) {
    if (attr != cudaFuncAttributeMaxDynamicSharedMemorySize || bytes != 60000) return 1;
    if (fails > 0) { fails--; return 2; }
    sets[f(0)][now]++;
    return 0;
}
"""

PROGRAM = """
#include "smem_optin.h"
#include <stdio.h>
#include <thread>
#include <vector>
thread_local int now = 0;
std::atomic<int> sets[3][70];
std::atomic<int> fails{0};
template <int K> int kernel(int) { return K; }
#define CHECK(x) do { if (!(x)) { printf("%s\\n", #x); return 1; } } while (0)
int main() {
    for (int i = 0; i < 3; i++) CHECK(allow_dynamic_smem<kernel<0>>(60000) == 0);
    CHECK(sets[0][0] == 1);
    now = 5;                                              // another device of the same process
    for (int i = 0; i < 3; i++) CHECK(allow_dynamic_smem<kernel<0>>(60000) == 0);
    CHECK(sets[0][5] == 1 && sets[0][0] == 1);
    now = 0;
    CHECK(allow_dynamic_smem<kernel<1>>(60000) == 0);     // another kernel of the same type
    CHECK(sets[1][0] == 1);
    now = 7;
    fails = 1;
    CHECK(allow_dynamic_smem<kernel<0>>(60000) == 2 && sets[0][7] == 0);
    CHECK(allow_dynamic_smem<kernel<0>>(60000) == 0 && sets[0][7] == 1);
    now = 66;                                             // beyond the mask: on every call
    for (int i = 0; i < 3; i++) CHECK(allow_dynamic_smem<kernel<0>>(60000) == 0);
    CHECK(sets[0][66] == 3);
    std::vector<std::thread> t;
    std::atomic<int> bad{0};
    for (int i = 0; i < 32; i++)
        t.emplace_back([&, i] {
            now = i % 4;
            for (int k = 0; k < 200; k++)
                if (allow_dynamic_smem<kernel<2>>(60000) != 0 || sets[2][now] < 1) bad++;
        });
    for (auto &x : t) x.join();
    CHECK(bad == 0);
    return 0;
}
"""


def test_once_per_kernel_and_device(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    (tmp_path / "main.cc").write_text(PROGRAM)
    exe = tmp_path / "main"
    subprocess.run([cxx, "-std=c++17", "-O2", "-pthread", f"-I{tmp_path}", f"-I{CSRC}", str(tmp_path / "main.cc"),
                    "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_every_launcher_uses_it():
    for f in os.listdir(CSRC):
        src = open(os.path.join(CSRC, f)).read()
        if f != "smem_optin.h":
            assert "cudaFuncSetAttribute" not in src and not re.search(r"static bool attr", src), f
