"""What a launch needs of a device -- the kernels' shared-memory limits, the
clusters it holds -- is set and asked for once for each device, whichever
context and host thread comes first (CPU only)."""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_01845_gb300", "csrc")

PROGRAM = r"""
#include "per_device.h"
#include <cstdio>
#include <thread>
#include <vector>

int main() {
    static wdc::PerDevice<int> value;
    std::atomic<int> made[2]{};
    std::atomic<int> wrong{0};
    std::vector<std::thread> threads;
    for (int t = 0; t < 16; ++t)
        threads.emplace_back([&, t] {
            for (int i = 0; i < 1000; ++i) {
                const int dev = (t + i) & 1;
                const int got = value.get(dev, [&](int& v) { ++made[dev]; v = 100 + dev; return true; });
                if (got != 100 + dev) ++wrong;
            }
        });
    for (auto& th : threads) th.join();
    // a value that may not be kept is made again, and handed out meanwhile
    static wdc::PerDevice<int> retried;
    int tries = 0;
    auto make = [&](int& v) { v = ++tries; return tries == 2; };
    const int a = retried.get(3, make), b = retried.get(3, make), c = retried.get(3, make);
    const int far = retried.get(1000, [](int& v) { v = 7; return true; });
    std::printf("%d %d %d %d %d %d %d\n", made[0].load(), made[1].load(), wrong.load(), a, b, c, far);
}
"""


def test_a_value_is_made_once_for_each_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "per_device.cpp", tmp_path / "per_device"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O2", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout
    assert out.split() == ["1", "1", "0", "1", "2", "2", "7"]


def test_no_launch_state_is_kept_for_the_process():
    """A function-local or file-level flag or count would hold for the first
    device alone, and be written by several threads."""
    kept = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.*h"))):
        for i, line in enumerate(open(path), 1):
            if re.match(r"\s*static\s+(?!constexpr|const\b)(bool|int|unsigned|size_t)\s+\w+(\[[^\]]*\])?\s*(=|\{|;)", line):
                kept.append(f"{os.path.basename(path)}:{i}: {line.strip()}")
    assert kept == []
