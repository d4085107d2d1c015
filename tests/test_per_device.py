"""Kernel attributes and occupancy answers belong to one device: what the library
keeps of them for the process (csrc/per_device.h) is kept per device."""
import glob
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1307_6720_gb300", "csrc")

PROGRAM = """
#include <atomic>
#include <cstdio>
#include <stdexcept>
#include <thread>
#include <vector>
#include "per_device.h"
#define NEED(c) if (!(c)) { std::printf("line %d\\n", __LINE__); return 1; }
int main() {
    mhs::PerDevice<const void*, int> p;
    int a = 0, b = 0, made = 0;
    auto make = [&] { return ++made; };
    NEED(p.get(0, &a, make) == 1 && p.get(0, &a, make) == 1);
    NEED(p.get(1, &a, make) == 2 && p.get(0, &b, make) == 3);      // another device, another kernel
    NEED(p.get(0, &a, make) == 1 && p.get(1, &a, make) == 2 && made == 3);
    bool threw = false;
    try { p.get(2, &a, []() -> int { throw std::runtime_error("refused"); }); } catch (const std::runtime_error&) { threw = true; }
    NEED(threw && p.get(2, &a, make) == 4);                         // nothing kept of the failure
    mhs::PerDevice<int, int> q;
    std::atomic<int> calls{0}, wrong{0};
    std::vector<std::thread> ts;
    for (int t = 0; t < 8; ++t)
        ts.emplace_back([&] {
            for (int r = 0; r < 1000; ++r)
                for (int d = 0; d < 4; ++d)
                    if (q.get(d, r % 5, [&] { ++calls; return 10 * d + r % 5; }) != 10 * d + r % 5) ++wrong;
        });
    for (auto& t : ts) t.join();
    NEED(calls == 20 && wrong == 0);
    return 0;
}
"""


def test_values_are_kept_per_device_and_made_once(tmp_path):
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_no_kernel_attribute_is_set_behind_a_flag_of_the_process():
    """A function-local flag or table would hold what the first device was told."""
    for path in glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")):
        text = open(path).read()
        assert not re.search(r"^[ \t]+static (thread_local )?(bool|int|std::map|std::set|std::once_flag|std::atomic)\b", text, re.M), path
