"""Kernel attributes belong to a device: a process with handles on two devices
sets them on both.  DeviceOnce (mg_optin.h) is compiled with the host compiler
against a stand-in for the runtime header, whose current device the test moves;
and every attribute that the sources set is set through it."""
import glob
import os
import re
import subprocess

from paper_1410_8568_gb300 import gbmg

CSRC = os.path.join(os.path.dirname(gbmg.__file__), "csrc")

RUNTIME = """
#pragma once
enum cudaError_t { cudaSuccess = 0, cudaErrorInvalidValue = 1, cudaErrorNoDevice = 100 };
extern int current;
inline cudaError_t cudaGetDevice(int *d) { *d = current; return current < 0 ? cudaErrorNoDevice : cudaSuccess; }
"""

PROGRAM = """
#include "mg_optin.h"
#include <stdio.h>
int current = 0;
int main()
{
    gbmg::DeviceOnce once;
    int runs = 0;
    bool fail = false;
    auto call = [&] { return once([&] { runs++; return fail ? cudaErrorInvalidValue : cudaSuccess; }); };
    auto show = [&](cudaError_t e) { printf("%d:%d ", runs, (int)e); };
    show(call()); show(call());                           // device 0: once
    current = 1; show(call()); show(call());              // device 1: once more
    current = 0; show(call());                            // device 0 is remembered
    current = 2; fail = true; show(call()); show(call()); // a failure is reported and tried again
    fail = false; show(call()); show(call());
    current = 70; show(call()); show(call());             // beyond the flags: every time
    current = -1; show(call());                           // no device
    return 0;
}
"""


def test_once_per_device(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    (tmp_path / "t.cpp").write_text(PROGRAM)
    exe = tmp_path / "t"
    subprocess.run(["g++", "-std=c++17", "-I", str(tmp_path), "-I", CSRC, str(tmp_path / "t.cpp"), "-o", str(exe)],
                   check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["1:0", "1:0", "2:0", "2:0", "2:0", "3:1", "4:1", "5:0", "5:0", "6:0", "7:0", "7:100"]


def test_every_attribute_is_set_through_it():
    found = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"\bcudaFuncSetAttribute\b", src):
            before = src[src.rfind("static ", 0, m.start()):m.start()]
            assert before.startswith("static DeviceOnce once;") and re.search(r"\bonce\(\s*\[", before), path
            found += 1
    assert found >= 6
