"""Kernel attributes are set once for every device, not once for the process.

Function attributes (the opt-in to large dynamic shared memory) and occupancy
belong to a device.  The helper that remembers them is host code: it is
compiled here on its own and called as contexts on several devices would.
"""
import os
import re
import shutil
import subprocess

import pytest

from paper_2306_00358_gb300 import build

PROGRAM = r"""
#include "per_device.h"
#include <cstdio>
#include <stdexcept>
#include <thread>
#include <vector>
int main() {
    trg::PerDevice p;
    int runs[3] = {0, 0, 0};
    for (int d : {0, 1, 0, 2, 1, 0})
        if (p.get(d, [&] { ++runs[d]; return 10 + d; }) != 10 + d) return 1;
    if (runs[0] != 1 || runs[1] != 1 || runs[2] != 1) return 2;
    trg::PerDevice q;      // a failure is tried again
    try { q.get(0, []() -> int { throw std::runtime_error("x"); }); return 3; } catch (const std::runtime_error&) {}
    if (q.get(0, [] { return 7; }) != 7) return 4;
    trg::PerDevice r;      // threads
    int count = 0;
    std::vector<std::thread> t;
    for (int i = 0; i < 8; ++i) t.emplace_back([&] { for (int k = 0; k < 100; ++k) r.get(k % 4, [&] { ++count; return 0; }); });
    for (auto& x : t) x.join();
    return count == 4 ? 0 : 5;
}
"""


def test_once_per_device(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host compiler")
    src = tmp_path / "p.cc"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-pthread", "-I", build.CSRC, str(src), "-o", str(tmp_path / "p")], check=True)
    assert subprocess.run([str(tmp_path / "p")]).returncode == 0


def test_no_kernel_attribute_is_set_once_per_process():
    for name in sorted(os.listdir(build.CSRC)):
        text = open(os.path.join(build.CSRC, name)).read()
        text = re.sub(r"//.*", "", text)
        for call in re.finditer(r"call_once\(", text):
            body = text[call.end():call.end() + 800].split("});")[0]
            assert "cudaFuncSetAttribute" not in body and "set_smem" not in body, name
            assert "Occupancy" not in body, name
