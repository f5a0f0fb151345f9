"""The per-device table that the kernel planners keep (csrc/per_device.h): a
second device is asked for its own number, although the first one's is known, and
a failed look-up is repeated."""
import os
import re
import subprocess

from paper_1902_10345_gb300 import build

SOURCE = r"""
#include <cassert>

#include "per_device.h"

int main() {
    sdfg::PerDevice<2> t;
    int asked[2] = {0, 0};
    auto find = [&](int device, int n) {
        return [&asked, device, n]() {
            ++asked[device];
            return n;
        };
    };
    for (int i = 0; i < 3; ++i) assert(t.get(0, 1, find(0, 4)) == 4);
    assert(asked[0] == 1 && asked[1] == 0);
    for (int i = 0; i < 3; ++i) assert(t.get(1, 1, find(1, 2)) == 2);
    assert(asked[0] == 1 && asked[1] == 1);
    assert(t.get(0, 1, find(0, 9)) == 4 && t.get(0, 0, find(0, 7)) == 7);
    assert(t.get(1, 0, find(1, 0)) == 0 && t.get(1, 0, find(1, 3)) == 3);
    return 0;
}
"""


def test_each_device_is_asked(tmp_path):
    src, exe = tmp_path / "per_device.cpp", tmp_path / "per_device"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-I" + build.CSRC, str(src), "-o", str(exe)], check=True)
    subprocess.run([str(exe)], check=True)


def test_no_table_without_a_device():
    """Occupancies and attributes hold for one device: no kernel source keeps numbers in a plain static array."""
    for name in sorted(os.listdir(build.CSRC)):
        if name.endswith((".cu", ".cuh")):
            text = open(os.path.join(build.CSRC, name), encoding="utf-8").read()
            assert not re.search(r"static (int|size_t|bool) \w+\[", text), name
