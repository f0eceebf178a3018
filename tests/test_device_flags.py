"""Set-up that belongs to a device: done once for each, kept when it succeeded (host only)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include "device_flags.h"
#include <cassert>
#include <thread>
#include <vector>
using namespace ckpt;
int main() {
    DeviceFlags flags;
    int calls[70] = {};
    auto visit = [&](int device, int rc) { return flags.once(device, [&] { ++calls[device]; return rc; }); };
    assert(visit(0, 0) == 0 && visit(0, 0) == 0 && calls[0] == 1);       // the second call on a device does nothing
    assert(visit(1, 0) == 0 && calls[1] == 1);                           // another device has work of its own
    assert(visit(2, -5) == -5 && visit(2, 0) == 0 && visit(2, 0) == 0 && calls[2] == 2);     // a failure is not kept
    assert(visit(63, 0) == 0 && visit(63, 0) == 0 && calls[63] == 1);
    assert(visit(69, 0) == 0 && visit(69, 0) == 0 && calls[69] == 2);    // beyond the table: every time
    DeviceFlags values;
    static int table[kMaxDevices];
    int found = 0, out = 0;
    auto find = [&](int* v) { ++found; *v = 7; return 0; };
    assert(values.once(3, table, &out, find) == 0 && out == 7);
    out = 0;
    assert(values.once(3, table, &out, find) == 0 && out == 7 && found == 1);
    DeviceFlags racing;
    static int shared[kMaxDevices];
    std::vector<std::thread> threads;
    for (int t = 0; t < 8; ++t)
        threads.emplace_back([&] {
            for (int i = 0; i < 20000; ++i) {
                int v = 0;
                assert(racing.once(i % 8, shared, &v, [&](int* o) { *o = i % 8 + 1; return 0; }) == 0 && v == i % 8 + 1);
            }
        });
    for (auto& t : threads) t.join();
}
"""


def test_once_per_device(tmp_path):
    source, program = tmp_path / "flags.cpp", tmp_path / "flags"
    source.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", os.path.join(ROOT, "paper_2502_12499_b200", "csrc"), str(source), "-o", str(program)], check=True)
    subprocess.run([str(program)], check=True, timeout=60)
