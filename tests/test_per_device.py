"""What the library asks a device about its kernels (attributes, resident clusters) is asked of every device, once, also
when the first calls come from several threads: the host header behind it, compiled with the host compiler."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "per_device.cuh"
#include <cstdio>
#include <thread>
#include <vector>

int main() {
    csd::PerDevice known;
    std::atomic<int> asked[csd::MAX_DEVICES] = {};
    std::atomic<int> wrong{0};
    std::vector<std::thread> threads;
    for (int t = 0; t < 8; ++t)
        threads.emplace_back([&] {
            for (int dev = 0; dev < csd::MAX_DEVICES; ++dev)
                for (int again = 0; again < 3; ++again)
                    if (known.get(dev, [&] { ++asked[dev]; return 10 * dev; }) != 10 * dev) ++wrong;
        });
    for (auto& t : threads) t.join();
    for (int dev = 0; dev < csd::MAX_DEVICES; ++dev)
        if (asked[dev] != 1) ++wrong;
    // a device outside the table is asked each time; a refusal is not kept
    int n = 0;
    csd::PerDevice other;
    for (int i = 0; i < 2; ++i)
        if (other.get(csd::MAX_DEVICES, [&] { return ++n; }) != i + 1) ++wrong;
    if (other.get(1, [] { return -1; }) != -1 || other.get(1, [] { return 4; }) != 4 || other.get(1, [] { return 5; }) != 4) ++wrong;
    std::printf("%d\n", (int)wrong);
    return wrong != 0;
}
"""


def test_every_device_is_asked_once(tmp_path):
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-pthread", "-I", os.path.join(ROOT, "paper_2312_11462_b200", "csrc"), "-o", str(exe), str(src)])
    assert subprocess.run([str(exe)], stdout=subprocess.PIPE, text=True, timeout=60).stdout == "0\n"


def test_no_attribute_of_a_kernel_is_settled_for_the_first_device_only():
    """Attributes belong to a kernel on one device: whoever sets one goes through PerDevice."""
    csrc = os.path.join(ROOT, "paper_2312_11462_b200", "csrc")
    for name in sorted(os.listdir(csrc)):
        lines = open(os.path.join(csrc, name)).read().split("\n")
        for i, line in enumerate(lines):
            if "cudaFuncSetAttribute(" in line:
                assert any(".get(dev," in before for before in lines[max(0, i - 8):i]), (name, i + 1)
