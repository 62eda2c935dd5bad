"""The truncation of the slice GEMMs' int64 sums (csrc/df_device.cuh), compiled for the host,
against its definition in Python's integers."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include "df_device.cuh"
#include <cstdio>
int main() {
  long long k;
  while (std::scanf("%lld", &k) == 1)
    for (int s = 0; s <= 8; ++s) std::printf("%d ", df::fixed_point_shift(s, k));
  return 0;
}
"""


def _shift(s, k):
    bound = sum((g + 1) * k << (14 + 8 * (s - 1 - g)) for g in range(s))
    return max(0, (bound - 1).bit_length() - 61) if bound else 0


def test_shift_equals_its_definition(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    (tmp_path / "cuda_runtime.h").write_text("#pragma once\n")
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "shift")
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", str(tmp_path), "-I", os.path.join(ROOT, "paper_2601_08077_gb300", "csrc"),
                    str(tmp_path / "main.cpp"), "-o", exe], check=True, capture_output=True, text=True)
    # every K near a power of two and near a switch of T, and the K ranges of both exchange GEMMs
    ks = sorted({1, 64, 128, 600, 1200, 1216, 15360, 32000, 2 ** 31 - 1}
                | {2 ** p + d for p in range(1, 40) for d in (-1, 0, 1)}
                | {(2 ** (61 + t) // sum((g + 1) << (14 + 8 * (s - 1 - g)) for g in range(s))) + d
                   for s in range(4, 9) for t in range(16) for d in (0, 1)} - {0})
    out = subprocess.run([exe], input=" ".join(map(str, ks)), capture_output=True, text=True, check=True).stdout.split()
    assert [int(v) for v in out] == [_shift(s, k) for k in ks for s in range(9)]
