"""Set-up of a kernel (dynamic shared memory, cluster sizes) belongs to one device, so it has to be made again on
every device a process uses: the helper that sees to it, with device numbers in place of devices, and that no
source file keeps such a set-up in a once-per-process static."""
import glob
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1905_08890_gb300", "csrc")

PROGRAM = r"""
#include <cstdlib>
#include <thread>
#include <vector>
#include "device_once.cuh"

int main()
{
    gr::DeviceOnce once;
    int calls[64] = {};
    const int order[] = {0, 1, 0, 40, 1, 31, 32, 40, 0, 31, 32};
    for (int d : order)
        if (once(d, [&] { calls[d]++; return d != 1; }) != (d != 1)) return 1;  // device 1's set-up fails, and stays so
    for (int d : {0, 1, 31, 32, 40})
        if (calls[d] != 1) return 2;
    gr::DeviceOnce shared;
    std::atomic<int> made[3] = {};
    std::vector<std::thread> t;
    for (int k = 0; k < 12; k++)
        t.emplace_back([&, k] {
            for (int r = 0; r < 1000; r++)
                if (!shared((k + r) % 3, [&] { made[(k + r) % 3]++; return true; })) std::_Exit(3);
        });
    for (auto &q : t) q.join();
    for (auto &m : made)
        if (m != 1) return 4;
    return 0;
}
"""


def test_once_on_each_device(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_kernel_attributes_are_set_per_device():
    """No attribute of a kernel is set by the initialiser of a static."""
    found = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        txt = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"cudaFuncSetAttribute", txt):
            found += 1
            before = txt[: m.start()]
            static = max(before.rfind("static const bool"), before.rfind("static const int"))
            assert before.rfind("per_device(") > static or "opt_in" in before[-400:], (path, before[-120:])
    assert found >= 8
