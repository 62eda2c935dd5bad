// Device helpers shared by the libdf kernels: integer-only FP64 bit
// manipulation (GB300's FP64 pipe is narrow, so the split and the
// recombination epilogues never touch it), and the balanced INT8 digit
// expansion of Section 3.2.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace df {

constexpr int kSMax = 8;            // digits per value
constexpr int kBlock = 128;         // auxiliary functions per block

// Truncation T of the int64 fixed-point sum of s slices and k products: |R| <= sum_g
// (g+1) k 2^14 2^(8(s-1-g)) must stay below 2^61 after dropping T low bits.  T = 0
// (exact) whenever that bound allows it.  In integers: a launch asks for nine of these,
// and on a host whose long double is emulated (Arm) they took 7 us of a call that way.
inline int fixed_point_shift(int s, long long k) {
  unsigned __int128 bound = 0;
  for (int g = 0; g < s; ++g) bound += ((unsigned __int128)(g + 1) * (unsigned __int128)k) << (14 + 8 * (s - 1 - g));
  int bits = 0;
  while (bits < 127 && ((unsigned __int128)1 << bits) < bound) ++bits;
  return bits > 61 ? bits - 61 : 0;
}

#ifdef __CUDACC__
// Row exponent from the bit pattern of max|row| (a non-negative double):
// the smallest e with vmax < 127/128 * 2^e; 0 for a zero row.
__device__ inline int exponent_from_max_bits_dev(uint64_t bits) {
  if (bits == 0) return 0;
  int E = (int)((bits >> 52) & 0x7FF);
  uint64_t m = bits & ((1ull << 52) - 1);
  if (E == 0) {
    int lz = __clzll((long long)m) - 11;
    m <<= lz;
    E = 1 - lz;
    m &= ((1ull << 52) - 1);
  }
  m |= (1ull << 52);
  return (E - 1023) + 1 + (m >= (127ull << 46) ? 1 : 0);
}

// Shifts of 64 and more give zero (PTX clamps the amount; in C++ they are undefined).
__device__ __forceinline__ uint64_t shr_clamped(uint64_t v, uint32_t k) {
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(k));
  return r;
}
__device__ __forceinline__ uint64_t shl_clamped(uint64_t v, uint32_t k) {
  uint64_t r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(k));
  return r;
}

// N = RNE(v * 2^(q1-e)) as int64, for |v| < 127/128 2^e and q1 <= 63.
// Integer-only, one path for every exponent: the significand at bits 62..10 moves right
// by k = 10 - (E - 1075 + q1 - e), which the headroom keeps >= 0; `out` holds what
// leaves it, so more than half (or half beside an odd quotient: the quotient's low
// bit goes to the bit of `out` that is always clear) rounds up.
__device__ __forceinline__ long long scaled_rne(uint64_t bits, int e, int q1 = 63) {
  const uint32_t hi = (uint32_t)(bits >> 32), lo = (uint32_t)bits;
  const int E = (int)((hi >> 20) & 0x7FFu);
  uint64_t m = ((uint64_t)((hi & 0xFFFFFu) | 0x100000u) << 42) | ((uint64_t)lo << 10);
  uint32_t k = (uint32_t)(1085 - q1 + e - E);
  if (E == 0) {  // zero, or subnormal (m 2^(1-1075)): its leading bit moves to bit 62
    m &= (1ull << 62) - 1;
    const int z = m ? __clzll((long long)m) - 1 : 0;
    m <<= z;
    k += (uint32_t)(z - 1);
  }
  uint64_t n = shr_clamped(m, k);
  const uint64_t out = shl_clamped(m, 64u - k) | (n & 1ull);
  n += out > (1ull << 63) ? 1ull : 0ull;
  return (hi >> 31) ? -(long long)n : (long long)n;
}

// Largest value over the TPR threads of a row (TPR = 32: one warp; TPR = 256: the
// whole block, through shared memory).
__device__ __forceinline__ uint32_t warp_max(uint32_t v) { return __reduce_max_sync(0xffffffffu, v); }
__device__ __forceinline__ uint64_t warp_max(uint64_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w > v ? w : v;
  }
  return v;
}
template <int TPR, typename T>
__device__ __forceinline__ T row_max(T m) {
  m = warp_max(m);
  if (TPR > 32) {
    __shared__ T part[TPR / 32];
    const int w = (threadIdx.x & (TPR - 1)) >> 5;
    if ((threadIdx.x & 31) == 0) part[w] = m;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < TPR / 32; ++i) m = part[i] > m ? part[i] : m;
  }
  return m;
}

// Row exponent of the values of a row: mh is this thread's largest high word
// (without the sign).  The high words settle it unless all are below the
// normal range, when the row is read again (bits(c): |value c|'s bits).
template <int TPR, typename Bits>
__device__ __forceinline__ int row_exponent(uint32_t mh, int lane, int cols, Bits bits) {
  mh = row_max<TPR>(mh);
  uint64_t m = (uint64_t)mh << 32;
  if (mh < 0x00100000u) {  // uniform over the row's threads
    m = 0;
    for (int c = lane; c < cols; c += TPR) {
      const uint64_t a = bits(c) & 0x7FFFFFFFFFFFFFFFull;
      m = a > m ? a : m;
    }
    m = row_max<TPR>(m);
  }
  return exponent_from_max_bits_dev(m);
}

// R to 53 bits, ties to even, for |R| < 2^61.
__device__ __forceinline__ long long round53(long long R) {
  const int hi = (int)(R >> 32);
  const uint32_t a = (uint32_t)(hi ^ (hi >> 31));  // |R|'s (or |R| - 1's) high word
  if (a >= (1u << 21)) {
    const int sh = 11 - __clz((int)a);  // bits to drop; exact powers of two have none set
    const long long lsb = (R >> sh) & 1;
    R += ((1ll << sh) >> 1) - 1 + lsb;
    R &= ~((1ll << sh) - 1);
  }
  return R;
}

// RNE(R 2^-r) for r >= 1, |R| < 2^61.
__device__ __forceinline__ long long rne_down(long long R, int r) {
  if (r >= 63) return 0;
  return (R + ((1ll << (r - 1)) - 1) + ((R >> r) & 1)) >> r;
}

// The X split's fast path for one element: N = RNE(fl64(r 2^k) 2^(63-g)), sh = k + 63 - g, for
// a row whose exponent bound is g.  kRound: |r| may have more than 53 bits.  top: the largest
// |N| so far (|N| - 1 of a negative one), its top 31 bits; lost: not zero once a shift pushed
// bits out of 64.
template <bool kRound>
__device__ __forceinline__ long long x_fixed(long long r, int sh, int &top, int &lost) {
  if (kRound) r = round53(r);
  const int hi = (int)(r >> 32);
  if ((unsigned)sh < 32u) {
    lost |= (hi >> (31 - sh)) ^ (hi >> 31);  // bits that the shift pushes out
    r <<= sh;
  } else if (sh < 0) {
    r = rne_down(r, -sh);
  } else {
    lost |= sh > 62 ? (int)(r != 0) : (int)((r >> (63 - sh)) != (r >> 63));
    r = sh > 62 ? 0 : r << sh;
  }
  const int h = (int)(r >> 32);
  top = max(top, h ^ (h >> 31));
  return r;
}

// Whether the bound g is the row's exponent and its N are right: attained (some |N| >= 2^62),
// no bits lost, and not within one unit of the 31 bits of 127/128 2^g.
__device__ __forceinline__ bool x_bound_is_exponent(int top, int lost) {
  return lost == 0 && top >= (1 << 30) && top < (127 << 24) - 1;
}

// Balanced digits of N: d[7..1] in [-128,127] from the bottom, d[0] the rest.
// Taking them from the bottom, digit k is ((N_k + 128) mod 256) - 128 and
// N_{k+1} = floor((N_k + 128) / 256), so with M = N + 128 (1 + 256 + ... +
// 256^6) every low digit is a plain byte of M minus 128 and the top digit is
// M >> 56 (arithmetic; |N| < 127 2^56 keeps M inside int64).
__device__ inline void balanced_digits(long long N, int d[kSMax]) {
  const long long M = N + 0x0080808080808080ll;
  d[0] = (int)(M >> 56);
#pragma unroll
  for (int t = 1; t < kSMax; ++t) d[t] = (int)((M >> (8 * (kSMax - 1 - t))) & 0xFF) - 128;
}

// Exact bf16 bit pattern of a small integer |d| <= 256 (no rounding needed).
// The float is formed as (1.5 2^23 + d) - 1.5 2^23: an integer add on the bit
// pattern (one ulp is 1 there) and one exact FP32 subtraction, both full-rate,
// instead of an int-to-float conversion.
__device__ inline uint16_t int_to_bf16_bits(int d) {
  const float f = __int_as_float(0x4B400000 + d) - 12582912.0f;
  return (uint16_t)(__float_as_uint(f) >> 16);
}

// Magnitude key of R 2^k (R != 0): |R| 2^k = M 2^(E - 64) with M normalised
// (top bit set).  Keys compare lexicographically (E, then M) like the exact
// magnitudes, and rounding to FP64 is monotone, so the largest |fl64(R 2^k)|
// of a row is the rounding of its largest key (ldexp_i64(M >> 1, E - 63):
// M's lowest bit is always zero).
__device__ inline void mag_key(long long R, int k, int &E, uint64_t &M) {
  const uint64_t u = R < 0 ? (uint64_t)(-(R + 1)) + 1ull : (uint64_t)R;
  const int lz = __clzll((long long)u);
  E = 64 - lz + k;
  M = u << lz;
}

// N = RNE(fl64(R 2^k) 2^(63-e)) as int64, where fl64 rounds to nearest even
// on 53 bits and flushes results below the normal range to zero exactly as
// ldexp_i64 does; the same value as scaled_rne(bits of ldexp_i64(R, k), e),
// in one pass of integer operations.  Requires |fl64(R 2^k)| < 127/128 2^e.
__device__ inline long long scaled_rne_i64(long long R, int k, int e) {
  if (R == 0) return 0;
  uint64_t u = R < 0 ? (uint64_t)(-(R + 1)) + 1ull : (uint64_t)R;
  const int nb = 64 - __clzll((long long)u);
  int ex = nb - 1 + k;  // exponent of the leading bit
  int sh1 = 0;
  if (nb > 53) {
    sh1 = nb - 53;
    uint64_t q = u >> sh1;
    const uint64_t rem = u & ((1ull << sh1) - 1);
    const uint64_t half = 1ull << (sh1 - 1);
    if (rem > half || (rem == half && (q & 1))) {
      q += 1;
      if (q == (1ull << 53)) {
        q >>= 1;
        sh1 += 1;
        ex += 1;
      }
    }
    u = q;
  }
  if (ex + 1023 <= 0) return 0;  // below the normal range: fl64 flushes to zero
  const int sh2 = sh1 + k + 63 - e;
  uint64_t n;
  if (sh2 >= 0) {
    n = u << sh2;
  } else {
    const int r = -sh2;
    if (r >= 64) {
      n = 0;
    } else {
      uint64_t q = u >> r;
      const uint64_t rem = u & ((1ull << r) - 1);
      const uint64_t half = 1ull << (r - 1);
      if (rem > half || (rem == half && (q & 1))) q += 1;
      n = q;
    }
  }
  return R < 0 ? -(long long)n : (long long)n;
}

// Correctly rounded fp64 of R * 2^k (R int64) by integer operations only.
// Results below the normal range are flushed to signed zero (never met:
// the scales of the DF tensors stay far from 2^-1022).
__device__ inline double ldexp_i64(long long R, int k) {
  if (R == 0) return 0.0;
  uint64_t sign = R < 0 ? (1ull << 63) : 0ull;
  uint64_t u = R < 0 ? (uint64_t)(-(R + 1)) + 1ull : (uint64_t)R;
  int nbits = 64 - __clzll((long long)u);
  uint64_t mant;
  int exp2 = nbits - 1 + k;  // value = 1.xxx * 2^exp2
  if (nbits <= 53) {
    mant = u << (53 - nbits);
  } else {
    int sh = nbits - 53;
    mant = u >> sh;
    uint64_t rem = u & ((1ull << sh) - 1);
    uint64_t half = 1ull << (sh - 1);
    if (rem > half || (rem == half && (mant & 1))) {
      mant += 1;
      if (mant == (1ull << 53)) {
        mant >>= 1;
        exp2 += 1;
      }
    }
  }
  int be = exp2 + 1023;
  if (be <= 0) return __longlong_as_double((long long)sign);
  if (be >= 2047) return __longlong_as_double((long long)(sign | (0x7FFull << 52)));
  uint64_t bits = sign | ((uint64_t)be << 52) | (mant & ((1ull << 52) - 1));
  return __longlong_as_double((long long)bits);
}

__device__ inline uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
#endif

}  // namespace df
