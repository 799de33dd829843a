"""Places of K's entries in the domains' dense blocks: every column of an internal row is an internal column of its
domain, one of its interface columns, or has no place (which pd_prefactor reports as a bad mesh)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_12484_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <vector>
#include "domain_rows.h"
int main() {   // in: columns, first, count, bnd_first, bnd_count, n_int, list length, list; out: the place of every column
    int nc, first, count, b0, nb, n_int, nl;
    while (std::scanf("%d %d %d %d %d %d %d", &nc, &first, &count, &b0, &nb, &n_int, &nl) == 7) {
        std::vector<int> bnd(nl + 1);
        for (int k = 0; k < nl; ++k)
            if (std::scanf("%d", &bnd[k]) != 1) return 1;
        for (int c = 0; c < nc; ++c) std::printf("%d ", pdg::domain_place(c, first, count, bnd.data(), b0, nb, n_int));
        std::printf("\n");
    }
}
"""


def test_every_column_has_its_place_or_none(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src = tmp_path / "t.cpp"
    src.write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(tmp_path / "t")], check=True)
    rng = np.random.default_rng(1)
    lines, want = [], []
    for n_dom, n_B in [(1, 0), (2, 5), (3, 1), (4, 40)]:
        counts = rng.integers(0, 6, n_dom)
        counts[0] = max(counts[0], 1)
        first = np.concatenate([[0], np.cumsum(counts)])
        lists = [np.sort(rng.choice(n_B, rng.integers(0, n_B + 1), replace=False)) for _ in range(n_dom)]
        off = np.concatenate([[0], np.cumsum([len(b) for b in lists])])
        n_int, flat = int(first[-1]), [int(j) for b in lists for j in b]
        for d in range(n_dom):
            lines.append(" ".join(map(str, [n_int + n_B, first[d], counts[d], off[d], len(lists[d]), n_int, len(flat), *flat])))
            place = {int(first[d]) + k: k for k in range(counts[d])}
            place |= {n_int + int(j): int(counts[d]) + k for k, j in enumerate(lists[d])}
            want.append([place.get(c, -1) for c in range(n_int + n_B)])
    out = subprocess.run([str(tmp_path / "t")], input="\n".join(lines), check=True, capture_output=True, text=True).stdout
    assert [[int(v) for v in row.split()] for row in out.splitlines()] == want


def test_kernels_report_an_entry_without_a_place():
    with open(os.path.join(CSRC, "k_dense64.cu")) as f:
        text = f.read()
    for kernel in ("k_assemble_rows", "k_domain_blocks"):
        body = text[text.index(f" {kernel}("):].split("\n}\n")[0]
        assert "ERR_NO_PLACE" in body, kernel
