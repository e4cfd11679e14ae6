"""The nuclear repulsion's pairs (csrc/pairs.cuh), compiled for the host: their number and the
pair of a given index at both ends of a row, up to the largest counts an int can name, against
Python's integers.  The pairs of 46342 nuclei no longer fit the int they were counted in."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <stdio.h>
#include "pairs.cuh"
int main() {
  long long n, t;
  while (scanf("%lld %lld", &n, &t) == 2) {
    int i, j;
    donof::pair_at(t, i, j);
    printf("%lld %d %d\n", donof::pair_count((int)n), i, j);
  }
}
"""


def test_counts_and_indices_of_pairs(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ unavailable")
    src, exe = tmp_path / "pairs.cpp", tmp_path / "pairs"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_2012_15662_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    rows = [1, 2, 3, 45, 46, 1448, 4096, 46340, 46341, 46342, 65536, 65537, 70000, 10**6, 2**31 - 2]
    asked = []
    for i in rows:
        for j in {0, i // 2, i - 1}:
            asked.append((i + 1, i * (i - 1) // 2 + j, i, j))
    out = subprocess.run([str(exe)], input="\n".join(f"{n} {t}" for n, t, _, _ in asked), capture_output=True, text=True,
                         check=True).stdout.split()
    got = [tuple(map(int, out[k:k + 3])) for k in range(0, len(out), 3)]
    assert got == [(n * (n - 1) // 2, i, j) for n, _, i, j in asked]
