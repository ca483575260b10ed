"""What a launch finds out once (function attributes, clusters that fit) is found out once per
GPU, also when several threads make their first calls together, and an error is not kept."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2607_03011_gb300", "csrc")

PROGRAM = r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"

int main() {
    isoloco::PerDevice d;
    std::atomic<int> made[2] = {{0}, {0}};
    std::atomic<bool> wrong{false};
    std::vector<std::thread> ts;
    for (int i = 0; i < 16; ++i)
        ts.emplace_back([&, i] {
            const int dev = i & 1;
            for (int k = 0; k < 1000; ++k) {
                int v = -1;
                const int e = d.get<int>(dev, &v, [&](int* x) { ++made[dev]; *x = 100 + dev; return 0; });
                if (e != 0 || v != 100 + dev) wrong = true;
            }
        });
    for (auto& t : ts) t.join();
    int v = -1, tries = 0;
    const int e1 = d.get<int>(5, &v, [&](int*) { ++tries; return 7; });
    const int e2 = d.get<int>(5, &v, [&](int* x) { ++tries; *x = 3; return 0; });
    const int ok5 = v;
    const int e3 = d.get<int>(1000, &v, [&](int* x) { *x = 9; return 0; });
    std::printf("%d %d %d | %d %d %d %d | %d %d\n", (int)wrong, (int)made[0], (int)made[1], e1, e2, ok5, tries, e3, v);
}
"""


def test_once_per_device(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.strip()
    assert out == "0 1 1 | 7 0 3 2 | 0 9"


def test_launchers_keep_nothing_for_the_whole_process():
    """No static flag or count stands in for a device's (a plan's kernels run on the plan's GPU)."""
    import re
    for name in os.listdir(CSRC):
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        assert not re.findall(r"\bstatic\s+(?:int|bool|size_t)\s+\w+\s*=\s*(?:0|false)\s*;", src), name
