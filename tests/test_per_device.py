"""The once-per-device set-up of the launchers (csrc/per_device.h) under host threads that launch at the
same time: a thread never sees the set-up done and its number missing.  Compiled with the thread
sanitizer, which reports any unordered access (the header needs no CUDA)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <thread>
#include <vector>
#include "per_device.h"

static int attribute[200];            // stands for the kernel's attribute on each device

int main() {
    for (int round = 0; round < 300; ++round) {
        auto* once = new loc::PerDevice;
        for (int& a : attribute) a = 0;
        std::vector<std::thread> ts;
        for (int t = 0; t < 8; ++t)
            ts.emplace_back([&, t] {
                for (int dev : {0, 63, 5}) {
                    int n = 0;
                    // one thread sets the attribute (setting it is the driver's business to order)
                    const int e = once->get(dev, &n, [&](int* v) {
                        if (t == 0) attribute[dev] = 152;
                        *v = 152;
                        return 0;
                    });
                    if (e != 0 || n != 152) std::exit(2);
                }
            });
        for (auto& t : ts) t.join();
        delete once;
    }
    // the attribute written before the number is seen by whoever sees the number
    for (int round = 0; round < 300; ++round) {
        auto* once = new loc::PerDevice;
        attribute[1] = 0;
        std::thread w([&] { int n = 0; once->get(1, &n, [](int* v) { attribute[1] = 7; *v = 9; return 0; }); });
        std::thread r([&] {
            int n = 0;
            while (once->get(1, &n, [](int*) { return 1; }) != 0) {}
            if (n != 9 || attribute[1] != 7) std::exit(3);
        });
        w.join();
        r.join();
        delete once;
    }
    // errors are passed on and not kept; devices past the slots are set up every time
    loc::PerDevice once;
    int n = 0, calls = 0;
    if (once.get(2, &n, [](int*) { return 11; }) != 11) return 4;
    if (once.get(2, &n, [](int* v) { *v = 3; return 0; }) != 0 || n != 3) return 5;
    for (int k = 0; k < 2; ++k)
        if (once.get(64, &n, [&](int* v) { ++calls; *v = 5; return 0; }) != 0 || n != 5) return 6;
    if (calls != 2) return 7;
    return 0;
}
"""


def test_threads_see_the_number_and_what_was_set_up(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    cmd = ["g++", "-std=c++17", "-O1", "-g", "-pthread", "-I", os.path.join(ROOT, "paper_1910_00572_gb300", "csrc")]
    built = subprocess.run(cmd + ["-fsanitize=thread", str(src), "-o", str(exe)], capture_output=True, text=True)
    if built.returncode != 0 and "tsan" in built.stderr:
        built = subprocess.run(cmd + [str(src), "-o", str(exe)], capture_output=True, text=True)   # no sanitizer here
    assert built.returncode == 0, built.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stderr[-2000:])
