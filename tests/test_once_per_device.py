"""The kernels' shared-memory opt-in is made on every device and by any host thread (csrc/dg_once.h):
the helper alone, compiled for the host, since a second GPU is not to be had in a test."""
import glob
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2305_13847_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "dg_once.h"
static dgm::OncePerDevice once;
int main() {
    int calls[100] = {};
    for (int pass = 0; pass < 3; ++pass)
        for (int d = 0; d < 100; ++d)
            if (once(d, [&] { return ++calls[d] == 1 && d == 2 ? 7 : 0; }) != (pass == 0 && d == 2 ? 7 : 0)) return 1;
    // once on each device, again after a failure (2), always beyond the array
    for (int d = 0; d < 100; ++d)
        if (calls[d] != (d >= 64 ? 3 : d == 2 ? 2 : 1)) return 2;
    dgm::OncePerDevice shared;
    std::atomic<int> n{0}, bad{0};
    std::vector<std::thread> t;
    for (int i = 0; i < 8; ++i)
        t.emplace_back([&] {
            for (int k = 0; k < 10000; ++k)
                if (shared(k % 4, [&] { ++n; return 0; }) != 0) ++bad;
        });
    for (auto &x : t) x.join();
    std::puts(bad == 0 && n >= 4 && n <= 32 ? "ok" : "bad");
    return 0;
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", (r.returncode, r.stdout)


def test_no_process_wide_flag_guards_a_device_attribute():
    for path in glob.glob(os.path.join(CSRC, "*")):
        text = open(path).read()
        if "cudaFuncSetAttribute" in text:
            assert not re.search(r"static\s+bool", text), path
