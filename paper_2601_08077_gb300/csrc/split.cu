// Split kernels (Section 3.2): FP64 values -> one power-of-two exponent per
// row (or column) and balanced signed 8-bit digits, most significant first.
//
//   e      = smallest integer with max|row| < 127/128 * 2^e   (0 for a zero row)
//   N      = RNE(v * 2^(63-e))  (|N| < 127 * 2^56)
//   digits = seven balanced bytes from the bottom, the rest on top, so that
//            v 2^(63-e) = sum_t d_t 256^(7-t), d_t in [-128, 127], |d_0| <= 127.
//
// All of it is integer arithmetic on the FP64 bit patterns.  The digits feed
// the tensor cores as BF16 (every integer in [-256, 256] is exact in BF16).
// These kernels are HBM-bound: each reads its FP64 input and writes s
// digits per value, in two passes over a row (its maximum, then the digits);
// for the B and C splits the second pass mostly hits L1/L2.  The X split's
// rows (128 functions x nocc values, up to 256 KB) take their exponent bound
// from the first GEMM and are read once.
#include "df_internal.h"

#include <climits>

namespace df {

namespace {

__device__ __forceinline__ uint64_t abs_bits(double v) {
  return (uint64_t)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
}

// Digit t of the balanced expansion of N as an exact FP32 value, from
// M = N + 128 (1 + 256 + ... + 256^6): the top digit is M >> 56, digit t >= 1
// is byte 7-t of M minus 128.  The FP32 is built as (1.5 2^23 + byte) - (1.5
// 2^23 + 128): one byte permute places the byte under the exponent bits and
// one FP32 subtraction is exact, so its top 16 bits are the digit's BF16.
__device__ __forceinline__ float digit_f32(long long M, int t) {
  if (t == 0) return __int_as_float(0x4B400000 + (int)(M >> 56)) - 12582912.0f;
  const uint32_t w = (7 - t) >= 4 ? (uint32_t)((unsigned long long)M >> 32) : (uint32_t)M;
  return __int_as_float((int)__byte_perm(w, 0x4B400000u, 0x7640u | (uint32_t)((7 - t) & 3))) - 12583040.0f;
}

// BF16 of two FP32 digits (exact) packed low, high.
__device__ __forceinline__ uint32_t bf16x2_of(float lo, float hi) {
  return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632u);
}

constexpr long long kDigitBias = 0x0080808080808080ll;  // 128 in each of the seven low bytes

// Four consecutive values of a row from column c on (zeros past cols); 16-byte
// loads when the row allows them.
template <bool kVec2>
__device__ __forceinline__ void load4(const double *__restrict__ row, int c, int cols, uint64_t (&v)[4]) {
  if (kVec2 && c + 4 <= cols) {
    const double2 a = __ldg(reinterpret_cast<const double2 *>(row + c));
    const double2 b = __ldg(reinterpret_cast<const double2 *>(row + c + 2));
    v[0] = (uint64_t)__double_as_longlong(a.x);
    v[1] = (uint64_t)__double_as_longlong(a.y);
    v[2] = (uint64_t)__double_as_longlong(b.x);
    v[3] = (uint64_t)__double_as_longlong(b.y);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = c + i < cols ? (uint64_t)__double_as_longlong(__ldg(row + c + i)) : 0ull;
  }
}

// Splits one row by TPR threads: its exponent, and s digits per value, four
// columns per thread and step (8-byte stores into rows of a multiple of 8
// digits, so columns past the row's end get zero digits).  nz (optional): the
// 64-wide column chunks in which this thread saw a nonzero, for cols <= 2048.
// The second pass reads the row from L1 or L2.
template <int TPR, bool kVec2>
__device__ __forceinline__ void split_row(const double *__restrict__ row, int cols, int lane, int nslices,
                                          int *__restrict__ exp, uint16_t *__restrict__ drow, long long plane_stride,
                                          uint32_t *nz) {
  uint32_t mh = 0u, bits = 0u;
#pragma unroll 4
  for (int c = 4 * lane; c < cols; c += 4 * TPR) {
    uint64_t v[4];
    load4<kVec2>(row, c, cols, v);
    uint32_t h[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = (uint32_t)(v[i] >> 32) & 0x7FFFFFFFu;
    mh = max(max(mh, max(h[0], h[1])), max(h[2], h[3]));
    if (nz && (h[0] | h[1] | h[2] | h[3] | (uint32_t)v[0] | (uint32_t)v[1] | (uint32_t)v[2] | (uint32_t)v[3]))
      bits |= 1u << ((c >> 6) & 31);
  }
  if (nz) *nz = bits;
  const int e = row_exponent<TPR>(
      mh, lane, cols, [&](int c) { return (uint64_t)__double_as_longlong(__ldg(row + c)); });
  if (lane == 0) *exp = e;
  for (int c = 4 * lane; c < cols; c += 4 * TPR) {
    uint64_t v[4];
    load4<kVec2>(row, c, cols, v);
    long long M[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) M[i] = scaled_rne(v[i], e) + kDigitBias;
#pragma unroll
    for (int t = 0; t < kSMax; ++t)
      if (t < nslices)
        *reinterpret_cast<uint2 *>(drow + (long long)t * plane_stride + c) =
            make_uint2(bf16x2_of(digit_f32(M[0], t), digit_f32(M[1], t)),
                       bf16x2_of(digit_f32(M[2], t), digit_f32(M[3], t)));
  }
}

// TPR threads per row (a warp, or the whole block for wide rows so that a
// few hundred rows of tens of thousands of columns still fill the GPU).
template <int TPR, bool kVec2>
__global__ void __launch_bounds__(256) split_rows_bf16_kernel(const double *__restrict__ A, long long rows,
                                                              int cols, long long ld, int nslices,
                                                              int *__restrict__ exps,
                                                              uint16_t *__restrict__ digits, long long dld,
                                                              long long plane_stride) {
  const int lane = threadIdx.x & (TPR - 1);
  const long long r = (long long)blockIdx.x * (blockDim.x / TPR) + (threadIdx.x / TPR);
  if (r >= rows) return;  // uniform over a row's threads (a whole block when TPR = 256)
  split_row<TPR, kVec2>(A + r * ld, cols, lane, nslices, exps + r, digits + r * dld, plane_stride, nullptr);
}

// Everything df_setup reads a dense B for, in one kernel: a CTA takes 32 rows
// of one B_P, compares them with the transposed tiles of B_P (an asymmetric B_P
// or a NaN sets *flag), splits them (a warp per row; with a permutation, output
// row (P', mu) reads input row (perm[P'], mu)), and ors each row's nonzero
// 64-wide column chunks into mask_mu[mu] (null past 2048 columns).  B comes from
// DRAM once: the transposed tiles and the second pass of a row are L2 and L1
// hits.  As three kernels (check, split, masks: one CTA per mu walking all P)
// the setup of 90 atoms (2.2 GB of B in, 3.3 GB of digits out) took 4.0 ms; this
// one took 2.0 with dependent tile loads, 1.55 with the next pair in flight
// (73% of the issue slots, 150 instructions a value) and 1.36 with the row maximum
// from the high words and a rounding without branches (5.4 TB/s of DRAM traffic:
// the strips in flight and their digits overflow L2, so part of B is read twice).
template <bool kVec2>
__global__ void __launch_bounds__(256) setup_rows_kernel(const double *__restrict__ B, int nao, int nslices,
                                                         int *__restrict__ exps, uint16_t *__restrict__ digits,
                                                         long long dld, long long plane_stride,
                                                         const int *__restrict__ perm,
                                                         uint32_t *__restrict__ mask_mu, int *__restrict__ flag) {
  __shared__ double tile[32][33];
  const int nt = (nao + 31) / 32;
  const int Pq = blockIdx.x / nt, bi = blockIdx.x - Pq * nt;
  const double *BP = B + (long long)(perm ? perm[Pq] : Pq) * nao * nao;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  bool bad = false;
  // tile (bi, bj) and its mirror (bj, bi): B[i][j] of the mirror must equal B[j][i]
  // = tile[lane][r].  The next pair's loads are in flight while one is compared.
  double a[4], m[4];
  const int i0 = bi * 32 + warp, jm = bi * 32 + lane;
  const double *pa = BP + (long long)i0 * nao + jm, *pm = pa;  // of the diagonal tile; each moves by a tile
  const long long row8 = 8ll * nao;
  auto load = [&](int bj) {
    const int j = bj * 32 + lane, im0 = bj * 32 + warp;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      a[k] = i0 + 8 * k < nao && j < nao ? __ldg(pa + k * row8) : 0.0;
      m[k] = im0 + 8 * k < nao && jm < nao ? __ldg(pm + k * row8) : 0.0;
    }
    pa += 32;
    pm += 4 * row8;
  };
  load(bi);
  for (int bj = bi; bj < nt; ++bj) {
    double c[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      tile[warp + 8 * k][lane] = a[k];
      c[k] = m[k];
    }
    if (bj + 1 < nt) load(bj + 1);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) bad |= !(c[k] == tile[lane][warp + 8 * k]);
    __syncthreads();
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(flag, 1);
  for (int r = warp; r < 32; r += 8) {
    const int mu = bi * 32 + r;
    if (mu >= nao) break;  // the whole warp
    const long long out = (long long)Pq * nao + mu;
    uint32_t nz = 0u;
    split_row<32, kVec2>(BP + (long long)mu * nao, nao, lane, nslices, exps + out, digits + out * dld, plane_stride,
                         mask_mu ? &nz : nullptr);
    if (mask_mu) {
      nz = __reduce_or_sync(0xffffffffu, nz);
      // the mask only gains bits: an old value at worst costs an atomic
      if (lane == 0 && (nz & ~*reinterpret_cast<volatile uint32_t *>(mask_mu + mu))) atomicOr(mask_mu + mu, nz);
    }
  }
}

// Rows of B from its packed layout (per P the upper triangle row by row,
// nao (nao + 1) / 2 values): output row r = (P', mu), P = perm[P'] (or P'),
// holds B_P mu nu for every nu (nu < mu read at the transposed position).
// One warp per row; the same two passes and digits as split_rows_bf16_kernel, two columns a
// lane (the transposed reads are a value each).  120 atoms, 600 AOs, six planes: the setup took
// 5.05 ms with the digits in arrays and a conversion each, 4.27 with their bytes placed in
// FP32; a screened chain of 60 atoms, whose zeros cost as much as any value since the rounding
// has no branches, 1.19 and 1.09.
__global__ void __launch_bounds__(256) split_rows_packed_kernel(const double *__restrict__ Bp, long long rows,
                                                                int nao, int nslices, int *__restrict__ exps,
                                                                uint16_t *__restrict__ digits, long long dld,
                                                                long long plane_stride,
                                                                const int *__restrict__ perm) {
  const int lane = threadIdx.x & 31;
  const long long r = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (r >= rows) return;
  const int Pq = (int)(r / nao), mu = (int)(r - (long long)Pq * nao);
  const int P = perm ? perm[Pq] : Pq;
  const double *BP = Bp + (long long)P * ((long long)nao * (nao + 1) / 2);
  const long long row_mu = (long long)mu * nao - (long long)mu * (mu - 1) / 2 - mu;  // + nu for nu >= mu
  auto at = [&](int nu) -> double {
    return nu >= mu ? __ldg(BP + row_mu + nu)
                    : __ldg(BP + (long long)nu * nao - (long long)nu * (nu - 1) / 2 + (mu - nu));
  };
  uint64_t m = 0;
  for (int c = lane; c < nao; c += 32) {
    const uint64_t a = abs_bits(at(c));
    m = a > m ? a : m;
  }
  m = warp_max(m);
  const int e = exponent_from_max_bits_dev(m);
  if (lane == 0) exps[r] = e;
  uint16_t *drow = digits + r * dld;
  // a pair past an odd row's end gets zero digits (rows of a multiple of 8 digits)
  for (int c = 2 * lane; c < nao; c += 64) {
    const uint64_t b1 = c + 1 < nao ? (uint64_t)__double_as_longlong(at(c + 1)) : 0ull;
    const long long M0 = scaled_rne((uint64_t)__double_as_longlong(at(c)), e) + kDigitBias;
    const long long M1 = scaled_rne(b1, e) + kDigitBias;
#pragma unroll
    for (int t = 0; t < kSMax; ++t)
      if (t < nslices)
        *reinterpret_cast<uint32_t *>(drow + (long long)t * plane_stride + c) =
            bf16x2_of(digit_f32(M0, t), digit_f32(M1, t));
  }
}

// One warp per row, int8 digits [nslices][rows][cols] (inspection entry point).
__global__ void split_rows_int8_kernel(const double *__restrict__ A, int rows, int cols, int ld, int nslices,
                                       int *__restrict__ exps, int8_t *__restrict__ digits) {
  const int lane = threadIdx.x & 31;
  const int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (r >= rows) return;
  const double *row = A + (long long)r * ld;
  uint64_t m = 0;
  for (int c = lane; c < cols; c += 32) {
    uint64_t a = abs_bits(row[c]);
    m = a > m ? a : m;
  }
  m = warp_max(m);
  const int e = exponent_from_max_bits_dev(m);
  if (lane == 0) exps[r] = e;
  for (int c = lane; c < cols; c += 32) {
    int d[kSMax];
    balanced_digits(scaled_rne((uint64_t)__double_as_longlong(row[c]), e), d);
    for (int t = 0; t < nslices; ++t) digits[((long long)t * rows + r) * cols + c] = (int8_t)d[t];
  }
}

// C [nrows][ncols] by columns: digits go to [t][c][r] (K-major).  A CTA takes 8
// columns with 512 threads, a warp 4 rows x 8 columns at a time (64-byte pieces
// of C's rows); all its loads are in flight before the first is used, and the
// values stay in registers between the maximum and the digits (up to 8 per
// thread, 512 rows; further rows are read again).  A warp per column walked them
// in two dependent passes (250 columns of 1200: 29 us).
// extra: words that the launches after it want set, the row bounds that the first
// exchange GEMM raises and the counters of the Coulomb passes.
constexpr int kColsT = 512;
constexpr int kColsHeld = 8;
__global__ void __launch_bounds__(kColsT) split_cols_bf16_kernel(const double *__restrict__ C, int nrows, int ncols,
                                                                 int nslices, int *__restrict__ exps,
                                                                 uint16_t *__restrict__ digits, long long dld,
                                                                 long long plane_stride, ColsExtra extra) {
  const int me = blockIdx.x * kColsT + threadIdx.x, all = gridDim.x * kColsT;
  for (int i = me; i < extra.nreset; i += all) extra.reset[i] = kRowBoundNone;
  for (int i = me; i < extra.nzero; i += all) extra.zero[i] = 0;
  const int c = blockIdx.x * 8 + (threadIdx.x & 7);
  const int r0 = threadIdx.x >> 3;
  constexpr int step = kColsT / 8;
  const bool col = c < ncols;
  uint64_t held[kColsHeld];
  uint64_t m = 0;
#pragma unroll
  for (int k = 0; k < kColsHeld; ++k) {
    const int r = r0 + k * step;
    held[k] = col && r < nrows ? (uint64_t)__double_as_longlong(__ldg(C + (long long)r * ncols + c)) : 0ull;
  }
#pragma unroll
  for (int k = 0; k < kColsHeld; ++k) {
    const uint64_t a = held[k] & 0x7FFFFFFFFFFFFFFFull;
    m = a > m ? a : m;
  }
  for (int r = r0 + kColsHeld * step; col && r < nrows; r += step) {
    const uint64_t a = abs_bits(__ldg(C + (long long)r * ncols + c));
    m = a > m ? a : m;
  }
#pragma unroll
  for (int o = 8; o < 32; o <<= 1) {
    const uint64_t w = __shfl_xor_sync(0xffffffffu, m, o);
    m = w > m ? w : m;
  }
  __shared__ uint64_t red[kColsT / 32][8];
  if ((threadIdx.x & 31) < 8) red[threadIdx.x >> 5][threadIdx.x & 7] = m;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kColsT / 32; ++w) m = red[w][threadIdx.x & 7] > m ? red[w][threadIdx.x & 7] : m;
  if (!col) return;
  const int e = exponent_from_max_bits_dev(m);
  if (r0 == 0) exps[c] = e;
  uint16_t *out = digits + (long long)c * dld;
  auto put = [&](uint64_t bits, int r) {
    int d[kSMax];
    balanced_digits(scaled_rne(bits, e), d);
#pragma unroll
    for (int t = 0; t < kSMax; ++t)
      if (t < nslices) out[(long long)t * plane_stride + r] = int_to_bf16_bits(d[t]);
  };
#pragma unroll
  for (int k = 0; k < kColsHeld; ++k)
    if (r0 + k * step < nrows) put(held[k], r0 + k * step);
  for (int r = r0 + kColsHeld * step; r < nrows; r += step)
    put((uint64_t)__double_as_longlong(__ldg(C + (long long)r * ncols + c)), r);
}

// The X split.  One CTA per (block b, row mu) of X [naux][nao][nocc] (nocc even):
// the row of the second exchange GEMM is X_b[mu, (P_local, i)], length nP*nocc,
// padded with zero digits up to a multiple of 64, one exponent per (block, mu).
//
// The first exchange GEMM leaves X as its exact int64 fixed-point sums R
// (Section 3.2's recombination before the final rounding); this kernel takes
// X = fl64(R 2^k), k = -14 - 8(s_b - 1) + T(s_b) + eC[i] + eB[(P, mu)], the
// one rounding of the emulated product, and splits it.  (Doing the rounding
// here keeps the GEMM's epilogue short.)
//
// The row's exponent needs its largest |X|.  The first GEMM recorded a bound g
// of it (the largest bitlen(|R|) + k of the row, rowE), so the exponent is g, or
// g + 1 when some |X| reaches 127/128 2^g.  The fast pass reads R once and
// writes the digits with e = g: N = RNE(X 2^(63-g)) is a left shift of R, after
// its rounding to 53 bits where it has more (kRound), for all but the elements
// far below the row's largest.  On the way it keeps the largest |N| (its top 31
// bits), which tells whether the bound is attained (|N| >= 2^62) and whether it
// is reached (|N| >= 127 2^56, to within one unit of the 31 bits), and whether a
// shift lost bits.  A row that is reached (about one in a hundred) or whose
// bound is not the row's takes the exact path (split_x_exact): it costs time
// only.
//
// The pass is bound by its integer instructions: with an exact key per element,
// a division per pair and plane offsets computed for a run-time slice count it
// took about 75 an element (120 atoms, 5 slices: 608 us for 2.4 GB).
constexpr int kSplitXThreads = 256;

struct XScale {
  const int *eB, *eC;  // (P, mu) row and orbital exponents of the first GEMM
  const int *s_blk;     // slices per block
  ShiftTable T;         // truncation of the first GEMM's fixed-point sum, by s
};

// One row of X as the split sees it: element (pl, i) is r[pl pstride + i] 2^(eP[pl] + eI[i]).
struct XRow {
  const long long *r;
  long long pstride;
  const int *eP, *eI;  // shared memory
  int nP, nocc, kpad;
};

// Exact path of a row: the exact magnitude keys of its elements (bit length +
// scale, then the normalised mantissa; rounding is monotone, so only the
// winning element is rounded), the exponent they give, then the digits.
// Returns the exponent.
__device__ __noinline__ int split_x_exact(const XRow x, int nslices, uint16_t *dst, long long plane) {
  __shared__ uint64_t red[kSplitXThreads / 32];
  __shared__ int redE[kSplitXThreads / 32];
  __shared__ int e_sh;
  const int klen = x.nP * x.nocc;
  int bE = INT_MIN;
  uint64_t bM = 0;
  for (int k = threadIdx.x; k < klen; k += kSplitXThreads) {
    const int pl = k / x.nocc, i = k - pl * x.nocc;
    const long long r = x.r[pl * x.pstride + i];
    if (r == 0) continue;
    int E;
    uint64_t M;
    mag_key(r, x.eP[pl] + x.eI[i], E, M);
    if (E > bE || (E == bE && M > bM)) {
      bE = E;
      bM = M;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const int E2 = __shfl_xor_sync(0xffffffffu, bE, o);
    const uint64_t M2 = __shfl_xor_sync(0xffffffffu, bM, o);
    if (E2 > bE || (E2 == bE && M2 > bM)) {
      bE = E2;
      bM = M2;
    }
  }
  if ((threadIdx.x & 31) == 0) {
    redE[threadIdx.x >> 5] = bE;
    red[threadIdx.x >> 5] = bM;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kSplitXThreads / 32; ++w)
      if (redE[w] > bE || (redE[w] == bE && red[w] > bM)) {
        bE = redE[w];
        bM = red[w];
      }
    // the row's largest |X| is the rounding of its largest exact magnitude
    const uint64_t top = bE == INT_MIN ? 0ull : abs_bits(ldexp_i64((long long)(bM >> 1), bE - 63));
    e_sh = exponent_from_max_bits_dev(top);
  }
  __syncthreads();
  const int e = e_sh;
  for (int k = threadIdx.x; k < x.kpad; k += kSplitXThreads) {
    int d[kSMax];
    long long N = 0;  // zero digits in the padding
    if (k < klen) {
      const int pl = k / x.nocc, i = k - pl * x.nocc;
      N = scaled_rne_i64(x.r[pl * x.pstride + i], x.eP[pl] + x.eI[i], e);
    }
    balanced_digits(N, d);
#pragma unroll
    for (int t = 0; t < kSMax; ++t)
      if (t < nslices) dst[(long long)t * plane + k] = int_to_bf16_bits(d[t]);
  }
  return e;
}

// S: digit planes written; kRound: some |R| may have more than 53 bits.
template <int S, bool kRound>
__global__ void __launch_bounds__(kSplitXThreads, 5)
    split_xblocks_kernel(const long long *__restrict__ R, int naux, int nao, int nocc, XScale xs,
                         const int *__restrict__ rowE, int *__restrict__ eX, uint16_t *__restrict__ Xd,
                         long long kb_ld, int nblk, RhoParts rp) {
  if (rp.part && blockIdx.y == 0) rho_from_parts(rp, blockIdx.x * kSplitXThreads + threadIdx.x, gridDim.x * kSplitXThreads);
  extern __shared__ int sh_e[];  // [kBlock] (P, mu) exponents + base, then [nocc] orbital exponents
  __shared__ int sh_top, sh_lost;
  const int mu = blockIdx.x;
  const int b = blockIdx.y;
  const int p0 = b * kBlock;
  const int nP = min(kBlock, naux - p0);
  int *eP = sh_e;
  int *eI = sh_e + kBlock;
  {
    const int s1 = xs.s_blk[b];
    const int kbase = -14 - 8 * (s1 - 1) + xs.T.v[s1];
    for (int q = threadIdx.x; q < nP; q += kSplitXThreads) eP[q] = kbase + xs.eB[(long long)(p0 + q) * nao + mu];
    for (int q = threadIdx.x; q < nocc; q += kSplitXThreads) eI[q] = xs.eC[q];
    if (threadIdx.x == 0) sh_top = sh_lost = 0;
  }
  const int g = __ldg(rowE + b * nao + mu);
  __syncthreads();
  const long long plane = (long long)nblk * nao * kb_ld;
  uint16_t *dst = Xd + ((long long)b * nao + mu) * kb_ld;
  const long long *row0 = R + ((long long)p0 * nao + mu) * nocc;  // element (pl, i) at row0[pl nao nocc + i]
  const long long pstride = (long long)nao * nocc;
  const int total = nP * (nocc >> 1);                    // pairs of neighbouring orbitals
  const int pairs = (nP * nocc + 63) / 64 * 32;          // and with the padding
  // far from the ends of the FP64 range: no |X| near 2^g overflows, and what
  // fl64 would flush to zero is below half a unit of N
  if (g > -900 && g < 1000) {
    const int hp = nocc >> 1;
    int pl = threadIdx.x / hp, ih = threadIdx.x - pl * hp;  // pair (pl, 2 ih)
    const int dpl = kSplitXThreads / hp, dih = kSplitXThreads - dpl * hp;
    uint32_t *out = reinterpret_cast<uint32_t *>(dst);
    const long long pl2 = plane >> 1;
    const int base = 63 - g;
    int top = 0, lost = 0;
    constexpr int kU = 2;  // pairs per thread in flight
    for (int q0 = threadIdx.x; q0 < pairs; q0 += kU * kSplitXThreads) {
      longlong2 v[kU];
      int sx[kU], sy[kU];
#pragma unroll
      for (int r = 0; r < kU; ++r) {
        v[r] = make_longlong2(0, 0);  // N = 0 (padding) gives zero digits
        sx[r] = sy[r] = 0;
        if (q0 + r * kSplitXThreads < total) {
          v[r] = *reinterpret_cast<const longlong2 *>(row0 + pl * pstride + 2 * ih);
          const int2 e2 = *reinterpret_cast<const int2 *>(eI + 2 * ih);
          sx[r] = base + eP[pl] + e2.x;
          sy[r] = base + eP[pl] + e2.y;
        }
        ih += dih;
        pl += dpl;
        if (ih >= hp) {
          ih -= hp;
          ++pl;
        }
      }
#pragma unroll
      for (int r = 0; r < kU; ++r) {
        const int q = q0 + r * kSplitXThreads;
        if (q >= pairs) break;
        const long long M0 = x_fixed<kRound>(v[r].x, sx[r], top, lost) + kDigitBias;
        const long long M1 = x_fixed<kRound>(v[r].y, sy[r], top, lost) + kDigitBias;
#pragma unroll
        for (int t = 0; t < S; ++t) out[q + t * pl2] = bf16x2_of(digit_f32(M0, t), digit_f32(M1, t));
      }
    }
    top = __reduce_max_sync(0xffffffffu, top);
    lost = __reduce_or_sync(0xffffffffu, lost);
    if ((threadIdx.x & 31) == 0) {
      atomicMax(&sh_top, top);
      if (lost) atomicOr(&sh_lost, lost);
    }
    __syncthreads();
    if (x_bound_is_exponent(sh_top, sh_lost)) {
      if (threadIdx.x == 0) eX[b * nao + mu] = g;
      return;
    }
    __syncthreads();  // every thread has read the verdict
  }
  const XRow x{row0, pstride, eP, eI, nP, nocc, 2 * pairs};
  const int e = split_x_exact(x, S, dst, plane);
  if (threadIdx.x == 0) eX[b * nao + mu] = e;
}

// K[mu][nu] = sum_b fl( 2^(eX[b,mu] + eX[b,nu] - 14 - 8(s_b - 1) + T(s_b)) * sum_sp R[b,sp] ),
// blocks in order (FP64), where R[b,sp][hi][lo] are the exact int64 partials of
// the second exchange GEMM (lower block-triangle, transposed) and the sum over
// the K splits of a block is exact.  A CTA takes a 32 x 8 tile of the lower
// triangle (rows hi, columns lo, so the partials are read along rows), four
// blocks' partials in flight, and writes both halves of K, the upper one through
// shared memory.  (One thread per element of the whole square read half of the
// partials column by column: 240 atoms 153 us.)
__global__ void __launch_bounds__(256) kpart_reduce_kernel(const long long *__restrict__ Rp,
                                                           const int *__restrict__ eX,
                                                           const int *__restrict__ s_blk, ShiftTable shiftT, int nao,
                                                           int nblk, int nsplit, double *__restrict__ K) {
  const int lo0 = blockIdx.x * 32, hi0 = blockIdx.y * 8;
  if (lo0 > hi0 + 7) return;  // above the diagonal
  const int lo = lo0 + (threadIdx.x & 31), hi = hi0 + (threadIdx.x >> 5);
  const long long bs = (long long)nao * nao;
  double acc = 0.0;
  if (hi < nao && lo <= hi) {
    const long long *src = Rp + (long long)hi * nao + lo;
    constexpr int kU = 4;
    for (int b0 = 0; b0 < nblk; b0 += kU) {
      long long R[kU];
      int k[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int b = b0 + u;
        R[u] = 0;
        k[u] = 0;
        if (b < nblk) {
          const int s = __ldg(s_blk + b);
          k[u] = __ldg(eX + b * nao + hi) + __ldg(eX + b * nao + lo) - 14 - 8 * (s - 1) + shiftT.v[s];
#pragma unroll 4
          for (int sp = 0; sp < nsplit; ++sp) R[u] += __ldg(src + ((long long)b * nsplit + sp) * bs);
        }
      }
#pragma unroll
      for (int u = 0; u < kU; ++u)
        if (b0 + u < nblk) acc += ldexp_i64(R[u], k[u]);
    }
    K[(long long)hi * nao + lo] = acc;
  }
  __shared__ double t[32][9];
  t[threadIdx.x & 31][threadIdx.x >> 5] = acc;
  __syncthreads();
  const int row = lo0 + (threadIdx.x >> 3), col = hi0 + (threadIdx.x & 7);
  if (row < nao && col < nao && row < col) K[(long long)row * nao + col] = t[threadIdx.x >> 3][threadIdx.x & 7];
}

}  // namespace

cudaError_t launch_split_rows_bf16(const double *A, long long rows, int cols, long long ld, int nslices,
                                   int *exps, uint16_t *digits, long long dld, long long plane_stride,
                                   cudaStream_t st) {
  if (rows <= 0) return cudaSuccess;
  const bool vec2 = (ld & 1) == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;
  const bool wide = cols >= kWideRow;
  const unsigned grid = (unsigned)(wide ? rows : (rows + 7) / 8);
  auto kern = wide ? (vec2 ? split_rows_bf16_kernel<256, true> : split_rows_bf16_kernel<256, false>)
                   : (vec2 ? split_rows_bf16_kernel<32, true> : split_rows_bf16_kernel<32, false>);
  kern<<<grid, 256, 0, st>>>(A, rows, cols, ld, nslices, exps, digits, dld, plane_stride);
  return cudaGetLastError();
}

cudaError_t launch_setup_rows(const double *B, int naux, int nao, int nslices, int *exps, uint16_t *digits,
                              long long dld, long long plane_stride, const int *perm, uint32_t *mask_mu, int *flag,
                              cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(flag, 0, sizeof(int), st);
  if (e == cudaSuccess && mask_mu) e = cudaMemsetAsync(mask_mu, 0, sizeof(uint32_t) * nao, st);
  if (e != cudaSuccess) return e;
  const bool vec2 = (nao & 1) == 0 && (reinterpret_cast<uintptr_t>(B) & 15) == 0;
  auto kern = vec2 ? setup_rows_kernel<true> : setup_rows_kernel<false>;
  kern<<<(unsigned)naux * (unsigned)((nao + 31) / 32), 256, 0, st>>>(B, nao, nslices, exps, digits, dld,
                                                                      plane_stride, perm, mask_mu, flag);
  return cudaGetLastError();
}

cudaError_t launch_split_rows_packed(const double *Bp, int naux, int nao, int nslices, int *exps, uint16_t *digits,
                                     long long dld, long long plane_stride, const int *perm, cudaStream_t st) {
  const long long rows = (long long)naux * nao;
  if (rows <= 0) return cudaSuccess;
  split_rows_packed_kernel<<<(unsigned)((rows + 7) / 8), 256, 0, st>>>(Bp, rows, nao, nslices, exps, digits, dld,
                                                                        plane_stride, perm);
  return cudaGetLastError();
}

cudaError_t launch_split_rows_int8(const double *A, int rows, int cols, int ld, int nslices, int *exps,
                                   int8_t *digits, cudaStream_t st) {
  if (rows <= 0) return cudaSuccess;
  split_rows_int8_kernel<<<(rows + 7) / 8, 256, 0, st>>>(A, rows, cols, ld, nslices, exps, digits);
  return cudaGetLastError();
}

cudaError_t launch_split_cols_bf16(const double *C, int nrows, int ncols, int nslices, int *exps,
                                   uint16_t *digits, long long dld, long long plane_stride, cudaStream_t st,
                                   const ColsExtra &extra) {
  if (ncols <= 0) return cudaSuccess;
  split_cols_bf16_kernel<<<(ncols + 7) / 8, kColsT, 0, st>>>(C, nrows, ncols, nslices, exps, digits, dld,
                                                             plane_stride, extra);
  return cudaGetLastError();
}

cudaError_t launch_split_xblocks(const long long *R, int naux, int nao, int nocc, int nslices, const int *eB,
                                 const int *eC, const int *s_blk, const ShiftTable &T1, const int *rowE,
                                 int *eX, uint16_t *Xd, long long kb_ld, int nblk, const RhoParts &rp,
                                 cudaStream_t st) {
  using Kern = void (*)(const long long *, int, int, int, XScale, const int *, int *, uint16_t *, long long, int,
                        RhoParts);
  // up to 4 slices a sum of nao products has at most 53 bits (2^(8(s-1) + 14) nao (1 + 2/256 + ...)) for
  // nao <= 2^14
  static const Kern exact[4] = {split_xblocks_kernel<1, false>, split_xblocks_kernel<2, false>,
                                split_xblocks_kernel<3, false>, split_xblocks_kernel<4, false>};
  static const Kern rounded[kSMax] = {split_xblocks_kernel<1, true>, split_xblocks_kernel<2, true>,
                                      split_xblocks_kernel<3, true>, split_xblocks_kernel<4, true>,
                                      split_xblocks_kernel<5, true>, split_xblocks_kernel<6, true>,
                                      split_xblocks_kernel<7, true>, split_xblocks_kernel<8, true>};
  if (nslices < 1 || nslices > kSMax || (nocc & 1)) return cudaErrorInvalidValue;
  const Kern kern = nslices <= 4 && nao <= 16000 ? exact[nslices - 1] : rounded[nslices - 1];
  const size_t sm = sizeof(int) * (size_t)(kBlock + nocc);
  if (sm > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
  }
  XScale xs{eB, eC, s_blk, T1};
  dim3 grid(nao, nblk);
  kern<<<grid, kSplitXThreads, sm, st>>>(R, naux, nao, nocc, xs, rowE, eX, Xd, kb_ld, nblk, rp);
  return cudaGetLastError();
}

cudaError_t launch_kpart_reduce(const long long *Rp, const int *eX, const int *s_blk, ShiftTable shiftT, int nao,
                                int nblk, int nsplit, double *K, cudaStream_t st) {
  dim3 grid((nao + 31) / 32, (nao + 7) / 8);
  kpart_reduce_kernel<<<grid, 256, 0, st>>>(Rp, eX, s_blk, shiftT, nao, nblk, nsplit, K);
  return cudaGetLastError();
}

}  // namespace df
