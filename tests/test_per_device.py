"""Kernel attributes belong to a device: a process that launches on a second one sets them there too.  The set-up class
of the launchers (csrc/fwime_device.h) runs here against a stand-in for cudaGetDevice, and every launcher that sets an
attribute goes through it."""
import glob
import os
import re
import subprocess

from paper_2206_02362_gb300 import build

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2206_02362_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "fwime_device.h"
static thread_local int device = 0;
static thread_local bool broken = false;
extern "C" cudaError_t cudaGetDevice(int *d)
{
    *d = device;
    return broken ? cudaErrorInvalidDevice : cudaSuccess;
}
static std::atomic<int> calls[70];
static int setup()
{
    static fwk::PerDevice<int> once;
    return once.get([] { calls[device]++; return 100 + device; });
}
int main()
{
    for (int d : {0, 1, 0, 3, 1, 63, 63, 64, 64}) {
        device = d;
        if (setup() != 100 + d) return 1;
    }
    std::vector<std::thread> t;
    for (int i = 0; i < 16; ++i) t.emplace_back([i] { device = 10 + i % 2; setup(); });
    for (auto &x : t) x.join();
    device = 1;
    broken = true;             // no current device: nothing is kept
    if (setup() != 101) return 2;
    for (int d : {0, 1, 3, 10, 11, 63, 64}) std::printf("%d ", (int)calls[d]);
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(PROGRAM)
    inc = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", inc, "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0
    # devices past the table are set up at every call, as when the device is not known
    assert r.stdout.split() == ["1", "2", "1", "1", "1", "1", "2"]


def test_launchers_set_attributes_per_device():
    sites = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        assert not re.search(r"static const \w+ \w+ =\s*(\[\] \{[^}]*)?cudaFuncSetAttribute", src), path
        sites += len(re.findall(r"static PerDevice<", src))
    assert sites == 5
