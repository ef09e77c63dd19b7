"""Kernel attributes belong to a device: the guard that sets them runs once on every
device, from any number of threads, and no source keeps a process-wide one (CPU)."""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1910_04727_gb300", "csrc")

PROGRAM = r"""
#include "once_per_device.h"
#include <atomic>
#include <thread>
#include <vector>
int main() {
    fm::OncePerDevice once;
    std::atomic<int> calls[5] = {};
    std::atomic<int> early{0};
    std::vector<std::thread> t;
    for (int k = 0; k < 40; ++k)
        t.emplace_back([&, k] {
            const int dev = k % 5;
            once.run(dev, [&] { std::this_thread::yield(); ++calls[dev]; });
            if (calls[dev] != 1) ++early;   // run() returned before the set-up was done
        });
    for (auto& x : t) x.join();
    for (auto& c : calls)
        if (c != 1) return 1;
    return early ? 2 : 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_runs_once_on_every_device(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    for _ in range(20):
        assert subprocess.run([str(exe)]).returncode == 0


def test_no_process_wide_guard_in_the_sources():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = open(path).read()
        assert "once_flag" not in text and "call_once" not in text, path
        assert not re.search(r"static bool \w+ = false;", text), path
