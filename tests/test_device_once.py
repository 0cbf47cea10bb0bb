"""Kernel attributes are set once per device, not once per process: the helper on the host, with device numbers
given by hand."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2011_10979_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "tvl1_device_once.h"
int main() {
    static tvl1::DeviceOnce once;
    int runs[66] = {}, bad = 0;
    std::mutex mu;
    auto use = [&](int d) {
        const int got = once.run(d, [&] { std::lock_guard<std::mutex> g(mu); return 100 + d + 0 * ++runs[d]; });
        if (got != 100 + d) ++bad;
    };
    std::vector<std::thread> th;
    for (int k = 0; k < 8; ++k) th.emplace_back([&, k] { for (int q = 0; q < 100; ++q) use((k + q) % 3); });
    for (auto &t : th) t.join();
    for (int k = 0; k < 3; ++k) use(65);
    printf("%d %d %d %d %d\n", runs[0], runs[1], runs[2], runs[65], bad);
}
"""


def test_every_device_is_prepared_once(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.check_call([cxx, "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)])
    assert subprocess.check_output([str(exe)], text=True).split() == ["1", "1", "1", "3", "0"]
