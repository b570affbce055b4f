"""The limit of dynamic shared memory that a kernel's launcher sets.

It holds for one device. The launchers' helper is compiled here against a fake
of the two runtime calls it makes: it has to set the limit once on every device
that launches, also from several threads at once, and again after a failure."""

import os
import re
import subprocess

from paper_2412_18379_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "launch_attr.h"

static thread_local int device = 0;
static std::atomic<int> sets[70];
static std::atomic<int> failures{0};
extern "C" cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute a, int bytes) {
    if (a != cudaFuncAttributeMaxDynamicSharedMemorySize || bytes != 100000) return cudaErrorInvalidValue;
    if (failures > 0) { --failures; return cudaErrorUnknown; }
    ++sets[device];
    return cudaSuccess;
}

int main() {
    static std::atomic<uint64_t> done{0};
    auto launch = [&](int d) { device = d; cs::allow_smem(done, nullptr, 100000); };
    for (int i = 0; i < 3; ++i) for (int d : {0, 1, 7, 63}) launch(d);
    for (int d : {0, 1, 7, 63}) if (sets[d] != 1) return 1;
    for (int i = 0; i < 3; ++i) launch(64);
    if (sets[64] != 3) return 2;
    failures = 1;
    for (int i = 0; i < 3; ++i) launch(2);
    if (sets[2] != 1 || failures != 0) return 3;
    std::atomic<int> unset{0};
    std::vector<std::thread> t;
    for (int i = 0; i < 8; ++i) t.emplace_back([&] { launch(5); unset += sets[5] == 0; });
    for (auto &x : t) x.join();
    if (unset || sets[5] < 1) return 4;
    const int before = sets[5];
    launch(5);
    return sets[5] == before ? 0 : 5;
}
"""


def test_the_limit_is_set_on_every_device(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", build.CSRC, "-I", build._cuda_inc(),
                    str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_no_launcher_sets_it_once_per_process():
    for f in sorted(os.listdir(build.CSRC)):
        if f.endswith(".cu"):
            text = open(os.path.join(build.CSRC, f)).read()
            assert not re.search(r"static bool \w+ = false;\s*if \(!\w+\) \{\s*cudaFuncSetAttribute", text), f
