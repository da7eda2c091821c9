"""Kernel attributes are set once per device, not once per process."""
import glob
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2410_19075_gb300", "csrc")

MAIN = r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"

int main()
{
    simk::PerDevice<int> done;
    std::atomic<int> calls{0};
    std::vector<std::thread> t;
    for (int k = 0; k < 16; ++k)
        t.emplace_back([&, k] {
            const int device = k % 4;
            if (done.get(device, [&] { ++calls; return 10 * device; }) != 10 * device) std::puts("wrong value");
        });
    for (auto &x : t) x.join();
    // one device's failure is its own
    std::printf("%d %d %d\n", calls.load(), done.get(7, [] { return -1; }), done.get(8, [] { return 0; }));
}
"""


def test_value_is_made_once_per_device(tmp_path):
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split() == ["4", "-1", "0"]


def test_no_attribute_is_set_under_a_process_wide_flag():
    """A flag of the process would leave every device but the first one without the attributes."""
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        for call in re.findall(r"call_once\((.*?)\);\n", open(path).read(), flags=re.S):
            assert "Attribute" not in call and "configure" not in call, (path, call)
