"""Kernel attributes are set on every device a process uses: the once-a-device helper against a fake
driver of several devices (no machine here has two GPUs), and no source that sets one only once a
process."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2102_03691_gb300", "csrc")

_PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <thread>
#include <vector>
#include "per_device.h"
enum Err { OK = 0, FAILED = 7 };
int main() {
    mhc::PerDevice once;
    std::atomic<int> calls[70] = {};
    bool fail = false;
    auto set = [&](int d) {
        return once(d, [&] { ++calls[d]; return fail ? FAILED : OK; });
    };
    auto check = [](bool ok, const char *what) { if (!ok) { std::printf("%s\n", what); std::exit(1); } };
    check(set(0) == OK && set(0) == OK && calls[0] == 1, "set once on a device");
    check(set(1) == OK && calls[1] == 1, "and on a second one");
    fail = true;
    check(set(2) == FAILED && set(0) == OK && calls[0] == 1, "a failure is returned");
    fail = false;
    check(set(2) == OK && set(2) == OK && calls[2] == 2, "and not kept");
    check(set(63) == OK && set(63) == OK && calls[63] == 1, "the last numbered device");
    check(set(64) == OK && set(64) == OK && calls[64] == 2, "beyond it every call sets");
    std::vector<std::thread> t;
    for (int q = 0; q < 8; ++q) t.emplace_back([&] { for (int d = 3; d < 60; ++d) if (set(d) != OK || !calls[d]) std::exit(2); });
    for (auto &x : t) x.join();
    const int before = calls[3];
    check(set(3) == OK && calls[3] == before, "after threads met on a device");
    return 0;
}
"""


def test_every_device_is_set_up_once(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src = tmp_path / "per_device.cpp"
    src.write_text(_PROGRAM)
    exe = tmp_path / "per_device"
    subprocess.run([cxx, "-std=c++17", "-Wall", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_no_attribute_is_set_once_a_process():
    for name in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, name)).read()
        assert not re.search(r"static\s+(?:const\s+)?(?:cudaError_t|bool)\s+\w+(?:\[\d\])?\s*=\s*[{(]?\s*(?:cudaFuncSetAttribute|false)", src), name
        # a function-local value that holds for the process and not for a device
        assert not re.search(r"static\s+int\s+\w+\s*=\s*-1\s*;", src), name
