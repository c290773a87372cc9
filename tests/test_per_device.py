"""A kernel's shared-memory limit belongs to a device: csrc/per_device.h raises it on each device that a process
uses, once, and again after a failure.  Compiled with the host compiler against a stand-in for the CUDA call."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2007_05540_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "per_device.h"
int main() {
    heff::PerDevice kernel, other;
    int raised[70] = {0}, fail = 0;
    auto on = [&](heff::PerDevice& k, int device) {
        return heff::once_per_device(k, device, [&] { ++raised[device]; return fail; });
    };
    for (int round = 0; round < 3; ++round)
        for (int device : {0, 1, 63}) if (on(kernel, device)) return 1;
    if (raised[0] != 1 || raised[1] != 1 || raised[63] != 1) return 2;      // once on each device
    if (on(other, 0) || raised[0] != 2) return 3;                            // and for each kernel
    fail = -5;
    if (on(kernel, 7) != -5 || on(kernel, 7) != -5 || raised[7] != 2) return 4;   // a failure is not remembered
    fail = 0;
    if (on(kernel, 7) || on(kernel, 7) || raised[7] != 3) return 5;
    if (on(kernel, 65) || on(kernel, 65) || raised[65] != 2) return 6;      // beyond the marks: every time
    std::puts("ok");
    return 0;
}
"""


def test_limit_is_raised_once_on_every_device(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout == "ok\n"


def test_no_process_wide_mark_is_left():
    """No launcher keeps "already raised" in a plain static of the process."""
    for f in os.listdir(CSRC):
        if f.endswith((".cu", ".cpp")):
            text = open(os.path.join(CSRC, f)).read()
            assert "static bool attr" not in text and "static bool done" not in text, f
