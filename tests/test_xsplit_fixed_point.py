"""The X split's one-pass digits and verdict (csrc/df_device.cuh), compiled for the host.

The split shifts a row's exact int64 sums R with scales k into N = RNE(fl64(R 2^k) 2^(63-g)), g the
bound that the first exchange GEMM recorded, and keeps the largest |N| and whether a shift lost
bits.  Where its verdict says that g is the row's exponent, exponent and every N must be the
oracle's; where it does not, the exact path recomputes the row, so the verdict may refuse but must
not do so for a row that is clear of the threshold.
"""
import math
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from oracle import df_oracle as O

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

STUB = r"""
#pragma once
#include <algorithm>
#include <cstdint>
#define __CUDACC__ 1
#define __device__
#define __forceinline__ inline
using std::max;
using std::min;
static inline int __clz(int v) { return v ? __builtin_clz((unsigned)v) : 32; }
static inline int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
static inline long long __double_as_longlong(double d) { long long v; __builtin_memcpy(&v, &d, 8); return v; }
static inline double __longlong_as_double(long long v) { double d; __builtin_memcpy(&d, &v, 8); return d; }
static inline float __int_as_float(int v) { float f; __builtin_memcpy(&f, &v, 4); return f; }
static inline uint32_t __float_as_uint(float f) { uint32_t v; __builtin_memcpy(&v, &f, 4); return v; }
static inline uint32_t __reduce_max_sync(unsigned, uint32_t v) { return v; }
static inline uint64_t __shfl_xor_sync(unsigned, uint64_t v, int) { return v; }
static inline void __syncthreads() {}
#define __shared__ static
static struct { unsigned x; } threadIdx;
"""

MAIN = r"""
#include "df_device.cuh"
#include <cstdio>
int main() {
  int round, count, g;
  while (std::scanf("%d %d %d", &round, &count, &g) == 3) {
    int top = 0, lost = 0;
    for (int i = 0; i < count; ++i) {
      long long r;
      int k;
      if (std::scanf("%lld %d", &r, &k) != 2) return 1;
      const int sh = k + 63 - g;
      std::printf("%lld ", round ? df::x_fixed<true>(r, sh, top, lost) : df::x_fixed<false>(r, sh, top, lost));
    }
    std::printf("%d\n", (int)df::x_bound_is_exponent(top, lost));
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("split")
    (d / "cuda_runtime.h").write_text(STUB)
    (d / "main.cpp").write_text('#include "cuda_runtime.h"\n' + MAIN)
    exe = str(d / "split")
    subprocess.run([gxx, "-O2", "-std=c++17", "-fwrapv", "-I", str(d), "-I", os.path.join(ROOT, "paper_2601_08077_gb300", "csrc"),
                    str(d / "main.cpp"), "-o", exe], check=True, capture_output=True, text=True)

    def run(rows):
        text = "\n".join("%d %d %d %s" % (rnd, len(Rs), g, " ".join("%d %d" % p for p in zip(Rs, ks)))
                         for rnd, Rs, ks, g in rows)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.splitlines()
        return [[int(v) for v in line.split()] for line in out]

    return run


def _bound(Rs, ks):
    """The first GEMM's: bit lengths, |R| - 1 for a negative R (one bit less for an exact power of two)."""
    b = [(R if R > 0 else -R - 1).bit_length() + k for R, k in zip(Rs, ks) if (R if R > 0 else -R - 1) != 0]
    return max(b) if b else None


def _rows(rng, count, most):
    """Rows whose largest elements lie around 127/128 2^g and around powers of two; |R| < 2^most."""
    rows = []
    for _ in range(count):
        Rs, ks = [], []
        for _ in range(int(rng.integers(1, 6))):
            nb = int(rng.integers(8, most + 1))
            mode = rng.random()
            unit = 2 ** max(0, nb - 54)
            if mode < 0.4:
                R = (127 << (nb - 7)) + int(rng.integers(-4, 5)) * unit
            elif mode < 0.5:
                R = (127 << (nb - 7)) + int(rng.integers(-4, 5)) * 2 ** max(0, nb - 31)
            elif mode < 0.7:
                R = 2 ** nb - 1 - int(rng.integers(0, 3)) * unit
            elif mode < 0.8:
                R = 2 ** (nb - 1)
            else:
                R = int(rng.integers(2 ** (nb - 1), 2 ** nb - 1, dtype=np.uint64))
            R = max(1, min(R, 2 ** most - 1))
            Rs.append(-R if rng.random() < 0.5 else R)
            # scales that spread the elements over a few digits, or far below the row's largest
            ks.append(int(rng.integers(-4, 5)) - nb if rng.random() < 0.8 else int(rng.integers(-140, -40)))
        rows.append((Rs, ks))
    return rows


@pytest.mark.parametrize("round53,most", [(1, 60), (0, 53)])
def test_verdict_and_digits(split, round53, most):
    rng = np.random.default_rng(most)
    rows = [(r, k, _bound(r, k)) for r, k in _rows(rng, 6000, most)]
    rows = [(r, k, g) for r, k, g in rows if g is not None]
    out = split([(round53, r, k, g) for r, k, g in rows])
    kept = 0
    for (Rs, ks, g), got in zip(rows, out):
        X = [math.ldexp(float(R), k) for R, k in zip(Rs, ks)]  # int -> float rounds to nearest even
        e = int(O.row_exponents(np.array([X]))[0])
        if got[-1]:
            kept += 1
            assert e == g, (Rs, ks)
            want = [int(round(Fraction(x) * Fraction(2) ** (63 - e))) for x in X]  # ties to even
            assert got[:-1] == want, (Rs, ks)
        else:
            # near the threshold (or at a negative power of two) only
            assert e != g or max(abs(x) for x in X) >= math.ldexp(127.0 / 128.0 - 2.0 ** -29, g), (Rs, ks)
    assert kept > len(rows) // 4
    # a bound one too high is the exponent only of a row that rounds up to its power of two
    for (Rs, ks, g), got in zip(rows, split([(round53, r, k, g + 1) for r, k, g in rows])):
        X = [math.ldexp(float(R), k) for R, k in zip(Rs, ks)]
        assert got[-1] == 0 or max(abs(x) for x in X) == math.ldexp(1.0, g), (Rs, ks)


def test_bound_one_too_low_is_refused(split):
    # a negative power of two: its recorded bound is one too low, |N| would be 2^63
    rows = [(1, [-(2 ** p), 3], [-p, -p - 2], _bound([-(2 ** p), 3], [-p, -p - 2])) for p in range(3, 60)]
    assert all(line[-1] == 0 for line in split(rows))
