"""Shared-memory limits of the kernels are raised on every device: the flag that says so is kept by device
(a handle on a second GPU would otherwise launch with the default limit).  Its bookkeeping, compiled for the
host, and that no launcher keeps a flag of the whole process instead."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0707_3405_gb300", "csrc")

PROGRAM = """
#include "device_once.h"
#include <initializer_list>
int main() {
    lg::DeviceOnce a, b;
    for (int d : {-1, 0, 1, 7, 63, 64, 1000}) if (a.done(d)) return 1;   // nothing done yet
    a.mark(0);
    if (!a.done(0) || a.done(1) || b.done(0)) return 2;                  // that device, that kernel
    a.mark(63);
    if (!a.done(0) || !a.done(63) || a.done(62)) return 3;
    for (int d : {-1, 64, 1000}) { a.mark(d); if (a.done(d)) return 4; } // without a bit: every time
    for (int d = 1; d < 63; ++d) if (a.done(d)) return 5;
    return 0;
}
"""


def test_flags_by_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_no_flag_of_the_whole_process():
    for f in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, f)).read()
        if "cudaFuncSetAttribute" in text:
            assert not re.search(r"static\s+std::atomic<bool>", text), f
