"""Per-device set-up (csrc/device_once.h): done once for each device, again
after a failure, by every thread that needs it; and no source keeps such state
per process or per thread instead."""
import glob
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1912_03278_gb300", "csrc")

PROGRAM = r"""
#include <cassert>
#include <thread>
#include <vector>
#include "device_once.h"
int main() {
    ihmc::DeviceOnce once;
    int calls[70] = {};
    auto set = [&](int dev, int result) { return once.run(dev, [&] { ++calls[dev]; return result; }); };
    assert(set(0, 0) == 0 && set(0, 0) == 0 && calls[0] == 1);
    assert(set(1, 7) == 7 && set(1, 0) == 0 && set(1, 0) == 0 && calls[1] == 2);   // a failure is tried again
    assert(set(63, 0) == 0 && set(63, 0) == 0 && calls[63] == 1);
    assert(set(65, 0) == 0 && set(65, 0) == 0 && calls[65] == 2);   // beyond the table: every time
    ihmc::DeviceValue v;
    assert(v.get(0, [] { return 0; }) == 0 && v.get(0, [] { return 152; }) == 152);
    assert(v.get(0, [] { return 1; }) == 152 && v.get(1, [] { return 80; }) == 80 && v.get(65, [] { return 9; }) == 9);
    ihmc::DeviceOnce shared;
    bool done[8] = {};
    std::vector<std::thread> ts;
    for (int t = 0; t < 8; ++t)
        ts.emplace_back([&, t] {
            bool mine = false;
            shared.run(t % 2, [&] { mine = true; return 0; });
            done[t] = mine;
        });
    for (auto &t : ts) t.join();
    assert((done[0] || done[2] || done[4] || done[6]) && (done[1] || done[3] || done[5] || done[7]));
    return 0;
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)])
    subprocess.check_call([str(exe)])


def test_no_process_wide_device_state():
    for f in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = open(f).read()
        assert not re.search(r"static\s+bool\s+\w+\s*=", text), f
        assert not re.search(r"static\s+thread_local\s+int\s+sms\b", text), f
