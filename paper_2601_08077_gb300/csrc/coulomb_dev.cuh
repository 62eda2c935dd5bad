// Device side of the Coulomb build (Section 2.1, Eqs. df-j-1 and df-j-2) shared
// by its own kernels (coulomb.cu) and by the slice GEMMs, whose spare warps run
// rho beside the first exchange GEMM and J beside the second (slicegemm.cu).
// Every rho_P and J_mn is summed in the same order wherever it is computed.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace df {

// A Coulomb pass as work items of one warp each, taken from a zeroed counter.
//   kind 1, rho: item 8 pg + w is part w of 8 of rho_P (rho_part) for the `group`
//   functions P = pg group .., written to part[w naux + P]; whoever runs next adds
//   the parts (rho_from_parts).
//   kind 2, J: item x + chunks y is 32 elements of the row pair (y, nao-1-y).
struct CoulombWork {
  int kind;             // 0 none, 1 rho, 2 J
  int naux, nao, packed, group, nitems;
  const double *B;
  const double *D;      // kind 1
  double *part;         // kind 1: [8][naux]
  const double *rho;    // kind 2
  double *J;            // kind 2
  int rows;             // kind 1: rho_part_rows
  const uint32_t *mask; // per mu the 64-wide nu chunks that hold a nonzero B_P mu nu (null: all)
  int *work;
};

// Sums of rho's parts to be done by a launch after the rho pass (null: none).
struct RhoParts {
  const double *part;
  double *rho, *rho2;   // rho2 optional
  int naux;
};

#ifdef __CUDACC__

// Start of row mu in a packed upper triangle of order nao.
__device__ __forceinline__ long long packed_row(int mu, int nao) {
  return (long long)mu * nao - (long long)mu * (mu - 1) / 2;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The strictly upper elements of B_P in row-pair order: pair q < nao/2 is
// row q from nu = q + 1 followed by row nao-1-q from nu = nao-q (nao - 1
// elements together, so every pair has the same length); for odd nao the
// middle row, q = nao/2, comes last alone.  Lane t of 256 takes the elements
// t, t + 256, ...: each warp reads 32 consecutive values of one row, and no
// lane has a per-row tail.
struct PairStream {
  int q, e;       // the current element: offset e in pair q
  int nao, L;     // L = nao - 1, the length of a full pair
  __device__ __forceinline__ void init(int j0, int n) {
    nao = n;
    L = n - 1;
    q = j0 / L;
    e = j0 - q * L;
  }
  __device__ __forceinline__ bool valid() const {
    return 2 * q + 1 < nao || (2 * q + 1 == nao && e < nao - 1 - q);
  }
  // (mu, nu), nu > mu, of the current element
  __device__ __forceinline__ void at(int &mu, int &nu) const {
    if (e < nao - 1 - q) {
      mu = q;
      nu = q + 1 + e;
    } else {
      mu = nao - 1 - q;
      nu = e + 1;
    }
  }
  __device__ __forceinline__ void advance(int step) {
    e += step;
    while (e >= L) {
      e -= L;
      ++q;
    }
  }
};

constexpr int kRhoLanes = 256;  // eight parts of a warp each

// Part w (lanes 32 w .. 32 w + 31 of kRhoLanes) of
//   rho_P = sum_mu B_P mu mu D_mu mu + 2 sum_{mu < nu} B_P mu nu D_mu nu
// for G functions P = P0 .. P0 + G-1 at once (the last one repeated past naux),
// in every lane.  The diagonal terms are spread over the lanes; the strictly
// upper ones stream in row-pair order, kQ steps of loads ahead of their FMAs,
// one load of D for G functions.  Offsets within the G functions are Off: 32 bits hold
// them while G nao^2 < 2^31 (kRho32Nao for one function), 64 for any nao.
constexpr int kRho32Nao = 46340;
template <bool kPacked, int G, int kQ, typename Off>
__device__ __forceinline__ void rho_part(const double *__restrict__ B, const double *__restrict__ D, int naux, int nao,
                                         int P0, int w, double (&v)[G]) {
  const int t = 32 * w + (threadIdx.x & 31);
  const Off n = nao;
  const Off stride = kPacked ? n * (n + 1) / 2 : n * n;
  const double *BP = B + (long long)P0 * stride;
  Off gs[G];
#pragma unroll
  for (int g = 0; g < G; ++g) gs[g] = G == 1 ? 0 : min(g, naux - 1 - P0) * stride;
  auto load = [&](Off idx, int g) -> double { return __ldg(BP + (G == 1 ? idx : idx + gs[g])); };
  auto index = [&](int mu, int nu) -> Off {
    const Off m = mu;
    return kPacked ? m * n - m * (m - 1) / 2 + (nu - mu) : m * n + nu;
  };
  double dia[G], off[G];
#pragma unroll
  for (int g = 0; g < G; ++g) dia[g] = off[g] = 0.0;
  for (int mu = t; mu < nao; mu += kRhoLanes) {
    const double d = __ldg(D + (long long)mu * nao + mu);
#pragma unroll
    for (int g = 0; g < G; ++g) dia[g] = fma(load(index(mu, mu), g), d, dia[g]);
  }
  const Off total = n * (n - 1) / 2;
  if (total > t) {
    PairStream ps;
    ps.init(t, nao);
    double bq[kQ][G], dq[kQ];
    auto fill = [&](int k) {
      dq[k] = 0.0;
#pragma unroll
      for (int g = 0; g < G; ++g) bq[k][g] = 0.0;
      if (ps.valid()) {
        int mu, nu;
        ps.at(mu, nu);
        const Off idx = index(mu, nu);
#pragma unroll
        for (int g = 0; g < G; ++g) bq[k][g] = load(idx, g);
        dq[k] = __ldg(D + (mu * n + nu));
      }
      ps.advance(kRhoLanes);
    };
#pragma unroll
    for (int k = 0; k < kQ; ++k) fill(k);
    const int mine = (int)((total - t + kRhoLanes - 1) / kRhoLanes);
    const int rounds = (mine + kQ - 1) / kQ;
    for (int r = 0; r < rounds; ++r) {
#pragma unroll
      for (int k = 0; k < kQ; ++k) {
#pragma unroll
        for (int g = 0; g < G; ++g) off[g] = fma(bq[k][g], dq[k], off[g]);
        fill(k);
      }
    }
  }
#pragma unroll
  for (int g = 0; g < G; ++g) v[g] = warp_sum(2.0 * off[g] + dia[g]);
}

// The same part for a B of mostly zero 64-wide chunks (nao <= 2048): rows mu = w,
// w + 8, ..., and of each the chunks set in its mask (null: all; a skipped term is
// an exact zero, so the bits are the same).  The row-pair stream would visit every
// element of the triangle to skip the zero ones (chain of 160 atoms, 2400
// functions of 800 AOs, 23% of the chunks: 1.36 ms; this one 0.50 ms by four
// functions, 0.94 ms with 32-wide windows of one function).
template <bool kPacked, int G>
__device__ __forceinline__ void rho_part_rows(const double *__restrict__ B, const double *__restrict__ D, int naux,
                                              int nao, const uint32_t *__restrict__ mask, int P0, int w,
                                              double (&v)[G]) {
  const int lane = threadIdx.x & 31;
  const int stride = kPacked ? nao * (nao + 1) / 2 : nao * nao;
  const double *BP = B + (long long)P0 * stride;
  int gs[G];
#pragma unroll
  for (int g = 0; g < G; ++g) gs[g] = G == 1 ? 0 : min(g, naux - 1 - P0) * stride;
  const uint32_t exist = nao > 64 * 31 ? ~0u : (1u << ((nao + 63) >> 6)) - 1u;
  double off[G];
#pragma unroll
  for (int g = 0; g < G; ++g) off[g] = 0.0;
  for (int mu = w; mu < nao; mu += kRhoLanes / 32) {
    uint32_t m = (mask ? __ldg(mask + mu) : ~0u) & exist & (~0u << (mu >> 6));
    const int row = kPacked ? mu * nao - mu * (mu - 1) / 2 - mu : mu * nao;
    for (; m; m &= m - 1u) {
      const int c0 = 64 * (__ffs((int)m) - 1) + lane;
      double b[2][G], d[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int nu = c0 + 32 * h;
        const bool in = nu >= mu && nu < nao;
#pragma unroll
        for (int g = 0; g < G; ++g) b[h][g] = in ? __ldg(BP + (G == 1 ? row + nu : row + nu + gs[g])) : 0.0;
        d[h] = in ? __ldg(D + (mu * nao + nu)) : 0.0;
        if (nu == mu) d[h] *= 0.5;  // off is counted twice
      }
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int g = 0; g < G; ++g) off[g] = fma(b[h][g], d[h], off[g]);
    }
  }
#pragma unroll
  for (int g = 0; g < G; ++g) v[g] = warp_sum(2.0 * off[g]);
}

// rho_P = its eight parts in order, by threads me, me + all, ...
__device__ __forceinline__ void rho_from_parts(const RhoParts &r, int me, int all) {
  for (int P = me; P < r.naux; P += all) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < kRhoLanes / 32; ++w) t += __ldg(r.part + (long long)w * r.naux + P);
    r.rho[P] = t;
    if (r.rho2) r.rho2[P] = t;
  }
}

// Element e of the row pair (y, nao-1-y): row y from column y, then row nao-1-y
// from its diagonal (nao + 1 elements per pair, one row alone in the middle
// when nao is odd).  False past the pair's end.
__device__ __forceinline__ bool pair_element(int nao, int y, int e, int &mu, int &nu) {
  const int m0 = y, m1 = nao - 1 - m0;
  const int len0 = nao - m0, len1 = m1 > m0 ? nao - m1 : 0;
  if (e >= len0 + len1) return false;
  mu = e < len0 ? m0 : m1;
  nu = e < len0 ? m0 + e : m1 + (e - len0);
  return true;
}

// sum_P B_P mu nu rho_P over ascending P, one FMA per P, kU loads of B ahead.
// kRing: kU loads always in flight, each taking the place of the one whose FMA was
// issued, for the few warps of a GEMM's helpers, whose FP64 pipe otherwise idles for
// a load's latency in every round (J beside the second GEMM: 188 -> 176 us at 60
// atoms, 435 -> 412 at 87).  The kernel of its own has warps enough to cover it and
// keeps the rounds (chain of 160 atoms, 1600 functions: 413 us, with the ring 449).
template <int kU, bool kRing>
__device__ __forceinline__ double coulomb_sum(const double *__restrict__ bp, long long stride,
                                              const double *__restrict__ rho, int naux) {
  double acc = 0.0;
  int P = 0;
  if constexpr (kRing) {
    if (naux >= kU) {
      double b[kU];
#pragma unroll
      for (int q = 0; q < kU; ++q) b[q] = __ldg(bp + q * stride);
      for (; P + 2 * kU <= naux; P += kU) {
        const double *next = bp + (P + kU) * stride;
#pragma unroll
        for (int q = 0; q < kU; ++q) {
          acc = fma(b[q], rho[P + q], acc);
          b[q] = __ldg(next + q * stride);
        }
      }
#pragma unroll
      for (int q = 0; q < kU; ++q) acc = fma(b[q], rho[P + q], acc);
      P += kU;
    }
  } else {
    for (; P + kU <= naux; P += kU) {
      double b[kU];
#pragma unroll
      for (int q = 0; q < kU; ++q) b[q] = __ldg(bp + (P + q) * stride);
#pragma unroll
      for (int q = 0; q < kU; ++q) acc = fma(b[q], rho[P + q], acc);
    }
  }
  for (; P < naux; ++P) acc = fma(__ldg(bp + P * stride), rho[P], acc);
  return acc;
}

// The next item of a counter, for all lanes of a warp.
__device__ __forceinline__ int take_item(int *work) {
  int v = 0;
  if ((threadIdx.x & 31) == 0) v = atomicAdd(work, 1);
  return v;
}
__device__ __forceinline__ int item_of_warp(int v) { return __shfl_sync(0xffffffffu, v, 0); }

// 32-bit offsets: rho_work makes groups of four up to nao = 16384, and df_build_JK runs a nao
// past kRho32Nao in order (64-bit ones beside them cost the GEMM's kernel 0.4 % of a step of
// 87 atoms without being taken).
template <bool kPacked, bool kRows, int G, int kQ>
__device__ __forceinline__ void rho_items(const CoulombWork &w) {
  int it = item_of_warp(take_item(w.work));
  while (it < w.nitems) {
    const int next = take_item(w.work);  // its latency passes beside this item
    const int P0 = (it >> 3) * G;
    double v[G];
    if constexpr (kRows)
      rho_part_rows<kPacked, G>(w.B, w.D, w.naux, w.nao, w.mask, P0, it & 7, v);
    else
      rho_part<kPacked, G, kQ, int>(w.B, w.D, w.naux, w.nao, P0, it & 7, v);
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
      for (int g = 0; g < G; ++g)
        if (P0 + g < w.naux) w.part[(long long)(it & 7) * w.naux + P0 + g] = v[g];
    }
    it = item_of_warp(next);
  }
}

__device__ __forceinline__ void coulomb_items(const CoulombWork &w) {
  const int nao = w.nao;
  const int chunks = (nao + 1 + 31) / 32;
  const long long stride = w.packed ? (long long)nao * (nao + 1) / 2 : (long long)nao * nao;
  for (;;) {
    const int it = item_of_warp(take_item(w.work));
    if (it >= w.nitems) break;
    const int y = it / chunks, x = it - y * chunks;
    int mu, nu;
    if (pair_element(nao, y, 32 * x + (int)(threadIdx.x & 31), mu, nu)) {
      const long long off = w.packed ? packed_row(mu, nao) + (nu - mu) : (long long)mu * nao + nu;
      double acc = 0.0;
      if (!w.mask || ((__ldg(w.mask + mu) >> (nu >> 6)) & 1u)) acc = coulomb_sum<16, true>(w.B + off, stride, w.rho, w.naux);
      w.J[(long long)mu * nao + nu] = acc;
      w.J[(long long)nu * nao + mu] = acc;
    }
    __syncwarp();
  }
}

template <bool kPacked, bool kRows>
__device__ __forceinline__ void rho_any_group(const CoulombWork &w) {
  if (w.group == 4)
    rho_items<kPacked, kRows, 4, 3>(w);
  else
    rho_items<kPacked, kRows, 1, 8>(w);
}

template <int kKind>
__device__ __forceinline__ void coulomb_work(const CoulombWork &w) {
  if constexpr (kKind == 1) {
    if (w.packed) {
      if (w.rows)
        rho_any_group<true, true>(w);
      else
        rho_any_group<true, false>(w);
    } else if (w.rows) {
      rho_any_group<false, true>(w);
    } else {
      rho_any_group<false, false>(w);
    }
  } else {
    coulomb_items(w);
  }
}
#endif

}  // namespace df
