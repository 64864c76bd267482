"""A kernel's dynamic shared-memory limit belongs to one device: it is raised once on each device that launches the
kernel (csrc/device_once.h, host code), a failure is not kept, and no other place sets it."""
import glob
import os
import re
import subprocess

from paper_0901_3512_gb300.build import CSRC

PROG = r'''
#include <cstdio>
#include <vector>
#include "device_once.h"
int main() {
    seedcg::DeviceOnce once;
    std::vector<int> on;
    auto set = [&](int d, bool fail) {
        try { once.run(d, [&]() { if (fail) throw 1; on.push_back(d); }); } catch (int) { on.push_back(-1); }
    };
    set(0, true);    // refused: tried again
    set(0, false);
    set(0, false);
    set(1, false);   // another device has its own
    set(0, false);
    set(1, false);
    set(99, false);  // past the table: every time
    set(99, false);
    for (int d : on) printf("%d ", d);
}
'''


def test_done_once_on_each_device_and_a_failure_is_not_kept(tmp_path):
    (tmp_path / "p.cpp").write_text(PROG)
    exe = str(tmp_path / "p")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(tmp_path / "p.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout
    assert out.split() == ["-1", "0", "1", "99", "99"]


def test_every_large_launch_goes_through_it():
    places = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for line in open(path).read().splitlines():
            if re.search(r"cudaFuncSetAttribute\(", line):
                places.append((os.path.basename(path), line.strip()))
    assert len(places) == 1 and places[0][0] == "internal.cuh" and "Kernel" in places[0][1], places
