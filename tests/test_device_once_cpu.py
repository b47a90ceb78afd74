"""The per-device attributes of the kernels (dynamic shared memory) are set on
every device, not on the first alone: DeviceOnce with a fake of the failing call."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2501_04776_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include "device_once.cuh"
int main() {
    iqp::DeviceOnce once;
    int calls[128] = {0}, fail = 0;
    auto on = [&](int d) { return once.run(d, [&] { ++calls[d]; return fail; }); };
    if (on(0) != 0 || on(0) != 0 || calls[0] != 1) return 1;   // once
    if (on(1) != 0 || calls[1] != 1) return 2;                 // and again on another device
    fail = 7;
    if (on(2) != 7 || on(0) != 0) return 3;                    // an error is returned ...
    fail = 0;
    if (on(2) != 0 || on(2) != 0 || calls[2] != 2) return 4;   // ... and tried again
    if (on(64) != 0 || on(64) != 0 || calls[64] != 2) return 5;
    if (on(63) != 0 || calls[63] != 1) return 6;
    std::thread t([&] { on(3); }), u([&] { on(4); });
    t.join();
    u.join();
    return calls[3] == 1 && calls[4] == 1 && on(3) == 0 && on(4) == 0 && calls[3] + calls[4] == 2 ? 0 : 7;
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-x", "c++", "-pthread", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_attributes_are_set_through_it():
    """The runtime call stands once, in the helper that takes a DeviceOnce."""
    uses = {f: len(re.findall(r"cudaFuncSetAttribute\(", open(os.path.join(CSRC, f)).read())) for f in sorted(os.listdir(CSRC))}
    assert {f: n for f, n in uses.items() if n} == {"common.cuh": 1}
