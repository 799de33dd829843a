"""Which elements take the SVD-free targets: strain_of compiled for the host
against its rule in FP64, just inside and just outside every bound (so that a
changed bound cannot leave the accuracy test of that path without cases)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from strain_cases import accepted, cases, gradients

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_12484_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include "proj3.cuh"
using namespace pdg::proj;
int main() {
    float A[9];
    while (std::fread(A, 4, 9, stdin) == 9) {
        float F[3][3];
        for (int i = 0; i < 9; ++i) F[i / 3][i % 3] = A[i];
        Strain S;
        std::printf("%d %d\n", (int)strain_of<true>(F, S), (int)strain_of<false>(F, S));
    }
}
"""


def test_the_path_takes_what_its_rule_says(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no CUDA compiler")
    src = tmp_path / "t.cu"
    src.write_text(HARNESS)
    subprocess.run([nvcc, "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(tmp_path / "t")], check=True,
                   capture_output=True)
    rng = np.random.default_rng(3)
    sig = cases()
    n = 20
    F = np.concatenate([gradients(rng, s, n) for s in sig])
    out = subprocess.run([str(tmp_path / "t")], input=F.tobytes(), check=True, capture_output=True).stdout
    took = np.array(out.split(), int).reshape(len(sig), n, 2)
    want = [accepted(s) for s in sig]
    assert 10 < sum(want) < len(sig) - 8
    for s, w, t in zip(sig, want, took):
        assert np.all(t == int(w)), (s, w)
