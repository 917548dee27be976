"""Per-device launch preparation (per_device.h): it runs once for every device,
the second one of a process too, and before any call for that device returns."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2405_14060_gb300", "csrc")
DRIVER = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
int main() {
    tn::PerDevice once;
    int runs[3] = {0, 0, 0};
    for (int dev : {0, 0, 1, 0, 1, 63, 63}) once.once(dev, [&] { ++runs[dev == 63 ? 2 : dev]; });
    if (runs[0] != 1 || runs[1] != 1 || runs[2] != 1) return 1;
    int far = 0;
    for (int i = 0; i < 2; ++i) once.once(64, [&] { ++far; });
    if (far != 2) return 2;
    tn::PerDevice shared;
    std::atomic<int> ready{0}, bad{0};
    std::vector<std::thread> ts;
    for (int t = 0; t < 8; ++t)
        ts.emplace_back([&, t] {
            shared.once(t & 1, [&] { ready |= 1 << (t & 1); });
            if (!(ready & (1 << (t & 1)))) ++bad;
        });
    for (auto &t : ts) t.join();
    return bad ? 3 : 0;
}
"""


def test_per_device_once(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "driver")
    r = subprocess.run([gxx, "-std=c++17", "-O2", "-pthread", "-I", CSRC, "-x", "c++", "-", "-o", exe],
                       input=DRIVER, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    assert subprocess.run([exe], timeout=60).returncode == 0
