"""Limits that belong to a device (the dynamic shared memory of a kernel): asked
for once on each device, not once per process."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_12484_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <initializer_list>
#include "per_device.h"
int main() {
    pdg::PerDevice known;
    int asked[80] = {};
    auto get = [&](int dev) { return known.get(dev, [&] { ++asked[dev < 0 ? 79 : dev]; return 1000 + dev; }); };
    for (int round = 0; round < 3; ++round)
        for (int dev : {0, 1, 63, 64, -1}) std::printf("%d ", get(dev));
    std::printf("\n%d %d %d %d %d\n", asked[0], asked[1], asked[63], asked[64], asked[79]);
}
"""


def test_each_device_is_asked_once(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src = tmp_path / "t.cpp"
    src.write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(tmp_path / "t")], check=True)
    values, asked = subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True).stdout.splitlines()
    assert values.split() == ["1000", "1001", "1063", "1064", "999"] * 3
    assert asked.split() == ["1", "1", "1", "3", "3"]      # (beyond the table: asked each time)


def test_no_limit_is_kept_per_process():
    """A function-local static is initialised once, on whichever device is current then."""
    for f in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, f)) as s:
            assert not re.search(r"\bstatic\b[^;{}]*=[^;{}]*(allow_max_dynamic_smem|cudaDeviceGetAttribute)", s.read()), f
