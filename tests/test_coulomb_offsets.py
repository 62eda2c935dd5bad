"""The element walk of the Coulomb pass rho (csrc/coulomb_dev.cuh), compiled for the host.

The header is compiled with g++ against a stub of the CUDA names it uses.  Loads go through a
stand-in of __ldg that never touches memory: it records the element's offset in B or D, so the
index arithmetic can be followed for tensors far larger than this machine holds (one B_P of
46342 functions is 17 GB).
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

STUB = r"""
#pragma once
#include <math.h>
#include <cstdint>
#include <algorithm>
#define __CUDACC__ 1
#define __device__
#define __forceinline__ inline
using std::min;
using std::max;
struct Idx { unsigned x; };
static Idx threadIdx;
double fake_ldg(const double *p);
static inline double __ldg(const double *p) { return fake_ldg(p); }
static inline uint32_t __ldg(const uint32_t *p) { return *p; }
static inline double __shfl_xor_sync(unsigned, double, int) { return 0.0; }
static inline int __shfl_sync(unsigned, int v, int) { return v; }
static inline void __syncwarp() {}
static inline int __ffs(int v) { return __builtin_ffs(v); }
static inline int atomicAdd(int *p, int v) { int o = *p; *p += v; return o; }
"""

MAIN = r"""
#include "coulomb_dev.cuh"
#include <cstdio>
#include <cstdlib>
#include <vector>

// addresses that are never dereferenced
static const double *const kB = reinterpret_cast<const double *>(1ull << 44);
static const double *const kD = reinterpret_cast<const double *>(1ull << 45);
static long long nB, nD, nao, naux, stride, P0;
static bool packed;
static long long bad, loadsB, loadsD;
static std::vector<int> *seen;  // per element of the group's B_P: visits (small cases)

double fake_ldg(const double *p) {
  const long long ob = p - kB, od = p - kD;
  if (p >= kB && ob < nB) {
    ++loadsB;
    if (seen) ++(*seen)[ob];
  } else if (p >= kD && od < nD) {
    ++loadsD;
    if (od % nao < od / nao) ++bad;  // below the diagonal
  } else {
    ++bad;
  }
  return 0.0;
}

template <bool kPacked, int G, int kQ, typename Off>
static void walk(int t) {
  double v[G];
  threadIdx.x = (unsigned)t;  // lane t % 32 of part t / 32
  df::rho_part<kPacked, G, kQ, Off>(kB, kD, (int)naux, (int)nao, (int)P0, t >> 5, v);
}

static long long upper(long long n) { return n * (n + 1) / 2; }

static void sizes(long long n, long long aux, bool pk) {
  nao = n;
  naux = aux;
  packed = pk;
  stride = pk ? upper(n) : n * n;
  nB = aux * stride;
  nD = n * n;
}

// every lane of a group of functions visits every upper element of each once
template <bool kPacked, int G, int kQ, typename Off>
static int cover(long long n, long long aux) {
  sizes(n, aux, kPacked);
  std::vector<int> visits(nB, 0);
  seen = &visits;
  for (P0 = 0; P0 < aux; P0 += G)
    for (int t = 0; t < 256; ++t) walk<kPacked, G, kQ, Off>(t);
  seen = nullptr;
  if (bad) return 1;
  for (long long P = 0; P < aux; ++P)
    for (long long m = 0; m < n; ++m)
      for (long long k = m; k < n; ++k) {
        const long long at = P * stride + (kPacked ? m * n - m * (m - 1) / 2 + k - m : m * n + k);
        // the group repeats the last function past naux
        const int want = P == aux - 1 ? 1 + (int)((G - aux % G) % G) : 1;
        if (visits[at] != want) return 2;
      }
  return 0;
}

// the lanes of a tensor of `n` functions that read the first and the last elements stay inside it
template <bool kPacked, typename Off>
static int large(long long n) {
  sizes(n, 2, kPacked);
  for (P0 = 0; P0 < 2; ++P0)
    for (int t : {0, 31, 255}) {
      loadsB = loadsD = bad = 0;
      walk<kPacked, 1, 8, Off>(t);
      const long long dia = (n - t + 255) / 256, off = (n * (n - 1) / 2 - t + 255) / 256;
      if (bad || loadsB != dia + off || loadsD != dia + off) {
        std::printf("n %lld packed %d P %lld t %d: out of range %lld, loads %lld and %lld of %lld\n", n, (int)kPacked, P0,
                    t, bad, loadsB, loadsD, dia + off);
        return 3;
      }
    }
  return 0;
}

int main(int argc, char **argv) {
  const long long n = std::atoll(argv[1]);
  if (n > 1000) {  // as the launches choose: 32 bits up to kRho32Nao, 64 for any size
    int r = large<false, long long>(n) | large<true, long long>(n);
    if (n <= df::kRho32Nao) r |= large<false, int>(n) | large<true, int>(n);
    return r;
  }
  for (long long aux : {1, 3, 6})
    if (int r = cover<false, 1, 8, int>(n, aux) | cover<true, 1, 8, int>(n, aux) | cover<false, 1, 8, long long>(n, aux) |
                cover<true, 1, 8, long long>(n, aux) | cover<false, 4, 3, int>(n, aux) | cover<true, 4, 3, int>(n, aux))
      return r;
  return 0;
}
"""


@pytest.fixture(scope="module")
def walker(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("walk")
    (d / "cuda_runtime.h").write_text(STUB)
    (d / "main.cpp").write_text('#include "cuda_runtime.h"\n' + MAIN)
    exe = str(d / "walk")
    # -fwrapv: 32-bit overflow wraps, as it does on the device
    subprocess.run([gxx, "-O2", "-std=c++17", "-fwrapv", "-I", str(d), "-I", os.path.join(ROOT, "paper_2601_08077_gb300", "csrc"),
                    str(d / "main.cpp"), "-o", exe], check=True, capture_output=True, text=True)
    return exe


# 46341^2 is the first square past 2^31, 65536^2 = 2^32; both parities of the row pairs
@pytest.mark.parametrize("nao", [1, 2, 3, 33, 64, 65, 258, 46340, 46341, 46342, 65537])
def test_rho_walk_stays_in_range(walker, nao):
    r = subprocess.run([walker, str(nao)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
