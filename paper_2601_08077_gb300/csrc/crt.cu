// CRT variant of the emulated FP64 GEMM: Ozaki scheme II (Ozaki, Uchino and
// Imamura, 2025), the INT8 alternative to slicing that Section 2.3 of the
// paper names, on the same tensor-core slice GEMM.  Section 4.5 of the paper
// notes that such a library takes a count of moduli rather than an accuracy;
// here the operand width q follows exactly from the moduli and K, so a level
// of Table 1 maps to a modulus count (df_crt_moduli_for_bits).
//
//   moduli   m_1 > m_2 > ... : integers <= 256 taken greedily downwards, each
//            coprime to the ones before; M = m_1 ... m_n < 2^128 (n <= 16)
//   width    q = the largest integer <= 63 with K 2^(2q-1) < M
//   operands e = smallest integer with max|row| < 127/128 2^e (0 for a zero
//            row); A' = RNE(A 2^(q-1-e)) per row, |A'| < 2^62
//   residues a_i = A' mod m_i in [-floor((m_i-1)/2), floor(m_i/2)] (BF16-exact)
//   GEMMs    S_i = a_i b_i^T exactly (products <= 2^14, FP32 chunks of 1024),
//            y_i = S_i mod m_i in the slice GEMM's epilogue (one byte each)
//   CRT      P' = the integer in (-M/2, M/2] with P' = y_i (mod m_i) for all i
//   result   fl64(P' 2^(e_r + f_c - 2(q-1))), one rounding to nearest even
//
// The residues come from the balanced base-256 digits of A' (the digits of the
// slice scheme): A' = sum_j b_j 256^j with signed bytes b_j, so A' mod m is
// congruent to two 4-way signed byte dot products (dp4a) with the centred
// weights 256^j mod m, a sum of at most 2^17 that FP32 reduces exactly.  The
// reconstruction accumulates sum_i y_i W_i (W_i the CRT weights) in 32-bit
// limbs, estimates the quotient by M in FP32 and finishes in 128-bit integers.
// No FP64 instruction is used: GB300's FP64 pipe is narrow.
#include "df_internal.h"

#include <cmath>
#include <cstring>

namespace df {

namespace {

struct CrtTab {
  int n;                            // moduli
  int q1;                           // q - 1
  int mod[kCrtMaxModuli];
  float modf[kCrtMaxModuli];
  float inv[kCrtMaxModuli];         // 1 / m
  int wlo[kCrtMaxModuli];           // centred 256^j mod m, j = 0..3, one signed byte each
  int whi[kCrtMaxModuli];           // j = 4..7
  uint32_t W[kCrtMaxModuli][4];     // CRT weights (M/m_i) ((M/m_i)^-1 mod m_i), 32-bit limbs
  uint32_t M[4];                    // product of the moduli, 32-bit limbs
  float f[4];                       // 2^(32k - sc), or 0 where a limb cannot matter
  float invM;                       // 2^sc / M
};

typedef unsigned __int128 u128;

int greedy_moduli(int n, int *out) {
  int k = 0;
  for (int m = 256; m >= 2 && k < n; --m) {
    bool ok = true;
    for (int j = 0; j < k && ok; ++j) {
      int a = m, b = out[j];
      while (b) {
        const int t = a % b;
        a = b;
        b = t;
      }
      ok = a == 1;
    }
    if (ok) out[k++] = m;
  }
  return k;
}

int bitlen128(u128 v) {
  int b = 0;
  while (v) {
    v >>= 1;
    ++b;
  }
  return b;
}

// q for K-term sums with n moduli (0 if the arguments admit none >= 2).
int operand_bits(long long K, int n) {
  if (K < 1 || K > (1ll << 26) || n < 2 || n > kCrtMaxModuli) return 0;
  int mods[kCrtMaxModuli];
  if (greedy_moduli(n, mods) != n) return 0;
  u128 M = 1;
  for (int i = 0; i < n; ++i) M *= (u128)mods[i];
  // K 2^(2q-1) < M  <=>  2^(2q-1) <= floor((M - 1) / K)  <=>  q <= bitlen / 2
  const u128 D = (M - 1) / (u128)K;
  int q = bitlen128(D) / 2;
  if (q > 63) q = 63;
  return q >= 2 ? q : 0;
}

bool make_tab(long long K, int n, CrtTab *t) {
  std::memset(t, 0, sizeof(*t));
  const int q = operand_bits(K, n);
  if (!q) return false;
  t->n = n;
  t->q1 = q - 1;
  greedy_moduli(n, t->mod);
  u128 M = 1;
  for (int i = 0; i < n; ++i) M *= (u128)t->mod[i];
  for (int i = 0; i < n; ++i) {
    const int m = t->mod[i];
    t->modf[i] = (float)m;
    t->inv[i] = 1.0f / (float)m;
    int lo = 0, hi = 0, w = 1 % m;
    for (int j = 0; j < 8; ++j) {
      const int c = w > m / 2 ? w - m : w;  // centred, in [-128, 127]
      if (j < 4)
        lo |= (c & 0xFF) << (8 * j);
      else
        hi |= (c & 0xFF) << (8 * (j - 4));
      w = (w * 256) % m;
    }
    t->wlo[i] = lo;
    t->whi[i] = hi;
    const u128 c = M / (u128)m;
    const int cm = (int)(c % (u128)m);
    int inv = 0;
    for (int x = 1; x < m; ++x)
      if ((cm * x) % m == 1) {
        inv = x;
        break;
      }
    const u128 Wi = c * (u128)inv;  // < M: c inv < (M / m) m
    for (int k = 0; k < 4; ++k) t->W[i][k] = (uint32_t)(Wi >> (32 * k));
  }
  for (int k = 0; k < 4; ++k) t->M[k] = (uint32_t)(M >> (32 * k));
  // scale the FP32 estimate of V = sum y_i W_i < 2^14 M so it stays below 2^100
  const int bl = bitlen128(M);
  const int sc = bl + 14 > 100 ? bl + 14 - 100 : 0;
  for (int k = 0; k < 4; ++k) {
    const int ex = 32 * k - sc;
    t->f[k] = (ex >= -126 && ex <= 127) ? std::ldexp(1.0f, ex) : 0.0f;
  }
  long double Ml = 0.0L;
  for (int k = 3; k >= 0; --k) Ml = Ml * 4294967296.0L + (long double)t->M[k];
  t->invM = (float)(std::ldexp(1.0L, sc) / Ml);
  return true;
}

// Centred residue, as an exact FP32 value, of the integer whose balanced digit
// words are (hi, lo), for an odd modulus: S = sum_j b_j (256^j mod m) has |S| <=
// 8 128^2 = 2^17, so the dot products started at the bits of 1.5 2^23 leave the
// FP32 1.5 2^23 + S; S - m rint(S / m) is then exact (S / m stays 1 / (2 m) > 2e-3
// away from a tie, its FP32 error is below 1e-4).  Six instructions where an
// integer Barrett step, the centring and the conversion to BF16 took 14.
__device__ __forceinline__ float residue_odd(int lo, int hi, const CrtTab &t, int i) {
  const float S = __int_as_float(__dp4a(lo, t.wlo[i], __dp4a(hi, t.whi[i], 0x4B400000))) - 12582912.0f;
  const float q = fmaf(S, t.inv[i], 12582912.0f) - 12582912.0f;
  return fmaf(-q, t.modf[i], S);
}

// The same for the modulus 256: the low digit, with 128 for -128.
__device__ __forceinline__ float residue_256(int lo) {
  const int b = (int)(signed char)(lo & 0xFF);
  return (float)(b == -128 ? 128 : b);
}

// TPR threads per row (a warp, or the whole block for wide rows): exponent,
// scaled integers, residue planes.  kInspect writes the residues as int16
// (inspection entry point), else BF16 bits.
template <bool kInspect, int TPR>
__global__ void __launch_bounds__(256)
    crt_split_rows_kernel(const double *__restrict__ A, long long rows, int cols, long long ld, const CrtTab t,
                          int *__restrict__ exps, uint16_t *__restrict__ planes, long long dld, long long pstride) {
  const int lane = threadIdx.x & (TPR - 1);
  const long long r = (long long)blockIdx.x * (blockDim.x / TPR) + (threadIdx.x / TPR);
  if (r >= rows) return;  // uniform over a row's threads
  const double *row = A + r * ld;
  const bool vec2 = (reinterpret_cast<uintptr_t>(row) & 15) == 0;
  uint32_t mh = 0u;
  auto bits = [&](int c) { return (uint64_t)__double_as_longlong(__ldg(row + c)); };
  auto high = [&](double v) { return (uint32_t)__double2hiint(v) & 0x7FFFFFFFu; };
  if (vec2) {
    for (int c = 2 * lane; c < cols; c += 2 * TPR) {
      const double2 v = c + 1 < cols ? __ldg(reinterpret_cast<const double2 *>(row + c)) : make_double2(__ldg(row + c), 0.0);
      mh = max(mh, max(high(v.x), high(v.y)));
    }
  } else {
    for (int c = lane; c < cols; c += TPR) mh = max(mh, high(__ldg(row + c)));
  }
  const int e = row_exponent<TPR>(mh, lane, cols, bits);
  if (lane == 0) exps[r] = e;
  uint16_t *drow = planes + r * dld;
  // four columns per lane per step: four independent chains per residue
  for (int c = 4 * lane; c < cols; c += 4 * TPR) {
    const int nv = cols - c < 4 ? cols - c : 4;
    int lo[4], hi[4];
    double x[4];
    if (vec2 && nv == 4) {
      const double2 u = __ldg(reinterpret_cast<const double2 *>(row + c));
      const double2 v = __ldg(reinterpret_cast<const double2 *>(row + c) + 1);
      x[0] = u.x, x[1] = u.y, x[2] = v.x, x[3] = v.y;
    } else {
      for (int h = 0; h < 4; ++h) x[h] = h < nv ? __ldg(row + c + h) : 0.0;
    }
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const uint64_t b = (uint64_t)__double_as_longlong(x[h]);
      // balanced digits: byte j of Mg is b_j + 128 for j < 7, the top byte is b_7
      const long long Mg = scaled_rne(b, e, t.q1) + 0x0080808080808080ll;
      lo[h] = (int)((uint32_t)Mg ^ 0x80808080u);
      hi[h] = (int)((uint32_t)((unsigned long long)Mg >> 32) ^ 0x00808080u);
    }
    // unrolled, so that the table entries are constant operands: indexed constant
    // loads were the kernel's limit (their unit 71% busy)
#pragma unroll
    for (int i = 0; i < kCrtMaxModuli; ++i) {
      if (i >= t.n) break;
      float res[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) res[h] = i == 0 ? residue_256(lo[h]) : residue_odd(lo[h], hi[h], t, i);
      uint16_t *dst = drow + (long long)i * pstride + c;
      // int16, or the BF16 of an exact small integer: its FP32's upper half
      uint32_t v[4];
#pragma unroll
      for (int h = 0; h < 4; ++h)
        v[h] = kInspect ? (uint32_t)(int)res[h] & 0xFFFFu : __float_as_uint(res[h]) >> 16;
      if (nv == 4 && ((reinterpret_cast<uintptr_t>(dst) & 7) == 0))
        *reinterpret_cast<uint2 *>(dst) =
            make_uint2(__byte_perm(v[0], v[1], 0x5410u), __byte_perm(v[2], v[3], 0x5410u));
      else
        for (int h = 0; h < nv; ++h) dst[h] = (uint16_t)v[h];
    }
  }
}

// P' from the residue bytes of one element (kParts K parts per modulus, added here: the
// sum is congruent, at most 255 kParts), then fl64(P' 2^k).  A loop over the moduli with the
// weights read by index, and the part count known to the compiler, so that the loads of
// several moduli are in flight: unrolled over all 16 moduli, with a loop over the parts
// inside, a load waited for the one before (2049 x 2049 of 12 moduli: 125 us, 78 this way; 16
// x 16: 8.0 and 4.2).
template <int kParts>
__device__ __forceinline__ double crt_value(const uint8_t *y, long long plane, const CrtTab &t, int k) {
  uint64_t a0 = 0, a1 = 0, a2 = 0, a3 = 0;  // V = sum_j a_j 2^(32j), each a_j < 2^46
  for (int i = 0; i < t.n; ++i) {
    uint64_t v = 0;
#pragma unroll
    for (int s = 0; s < kParts; ++s) v += y[(i * kParts + s) * plane];
    a0 += v * t.W[i][0];
    a1 += v * t.W[i][1];
    a2 += v * t.W[i][2];
    a3 += v * t.W[i][3];
  }
  // V / M < 2^14; the FP32 estimate is within 1/64 of it, so floor is off by at most 1
  const float vf = (float)a0 * t.f[0] + (float)a1 * t.f[1] + (float)a2 * t.f[2] + (float)a3 * t.f[3];
  const long long qe = (long long)__float2int_rd(vf * t.invM);
  // R = V - qe M in 128-bit two's complement (it lies in (-M, 2M))
  const u128 R0 = (u128)(long long)((long long)a0 - qe * (long long)t.M[0]) +
                  ((u128)(long long)((long long)a1 - qe * (long long)t.M[1]) << 32) +
                  ((u128)(long long)((long long)a2 - qe * (long long)t.M[2]) << 64) +
                  ((u128)(long long)((long long)a3 - qe * (long long)t.M[3]) << 96);
  __int128 R = (__int128)R0;
  const __int128 M = (__int128)(((u128)t.M[3] << 96) | ((u128)t.M[2] << 64) | ((u128)t.M[1] << 32) | (u128)t.M[0]);
  if (R < 0)
    R += M;
  else if (R >= M)
    R -= M;
  if (2 * R > M) R -= M;  // the representative in (-M/2, M/2]
  if (R == 0) return 0.0;
  const bool neg = R < 0;
  const u128 u = neg ? (u128)(-R) : (u128)R;
  const uint64_t hi = (uint64_t)(u >> 64), lo = (uint64_t)u;
  if (hi == 0 && lo < (1ull << 63)) return ldexp_i64(neg ? -(long long)lo : (long long)lo, k);
  // 63 leading bits plus a sticky bit: rounding them once gives the rounding of u
  const int nb = hi ? 128 - __clzll((long long)hi) : 64;
  const int sh = nb - 63;
  uint64_t win = (uint64_t)(u >> sh);
  if (u & (((u128)1 << sh) - 1)) win |= 1ull;
  return ldexp_i64(neg ? -(long long)win : (long long)win, k + sh);
}

template <int kParts>
__global__ void __launch_bounds__(256)
    crt_reconstruct_kernel(const uint8_t *__restrict__ Y, int M, int N, long long ldy, long long plane,
                           const int *__restrict__ ea, const int *__restrict__ eb, const CrtTab t,
                           double *__restrict__ out, long long ldo) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  const int ebn = eb[n];
  for (int m = blockIdx.y; m < M; m += gridDim.y)
    out[(long long)m * ldo + n] = crt_value<kParts>(Y + (long long)m * ldy + n, plane, t, ea[m] + ebn - 2 * t.q1);
}

// The same for a Gram matrix, whose residues exist in the 128-wide tiles (i, j >= i):
// a CTA takes 8 rows m0 .. of the columns n0 .. n0 + 31 >= m0 and writes them and
// their transpose (64-byte pieces); a value is a chain of a few hundred integer
// instructions, so the tile is one value per thread.
template <int kParts>
__global__ void __launch_bounds__(256)
    crt_reconstruct_sym_kernel(const uint8_t *__restrict__ Y, int N, long long ldy, long long plane,
                               const int *__restrict__ ea, const CrtTab t, double *__restrict__ out, long long ldo) {
  __shared__ double tile[32][9];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n0 = blockIdx.x * 32, n = n0 + lane;
  const int en = n < N ? ea[n] : 0;
  const int last = min(N, n0 + 32);
  for (int m0 = blockIdx.y * 8; m0 < last; m0 += gridDim.y * 8) {
    const int m = m0 + warp;
    if (m < N && n < N) {
      const double v = crt_value<kParts>(Y + (long long)m * ldy + n, plane, t, ea[m] + en - 2 * t.q1);
      out[(long long)m * ldo + n] = v;
      tile[lane][warp] = v;
    }
    if (m0 >= n0) continue;  // beside the diagonal both triangles are computed; m0 only grows
    __syncthreads();
    const int r = threadIdx.x >> 3, c = threadIdx.x & 7;  // m0 + c < n0 <= N - 1
    if (n0 + r < N) out[(long long)(n0 + r) * ldo + m0 + c] = tile[r][c];
    __syncthreads();
  }
}

cudaError_t launch_crt_split(const double *A, long long rows, int cols, long long ld, const CrtTab &t, int *exps,
                             uint16_t *planes, long long dld, long long pstride, bool inspect, cudaStream_t st) {
  if (rows <= 0) return cudaSuccess;
  if (cols >= kWideRow) {
    const dim3 grid((unsigned)rows);
    if (inspect)
      crt_split_rows_kernel<true, 256><<<grid, 256, 0, st>>>(A, rows, cols, ld, t, exps, planes, dld, pstride);
    else
      crt_split_rows_kernel<false, 256><<<grid, 256, 0, st>>>(A, rows, cols, ld, t, exps, planes, dld, pstride);
  } else {
    const dim3 grid((unsigned)((rows + 7) / 8));
    if (inspect)
      crt_split_rows_kernel<true, 32><<<grid, 256, 0, st>>>(A, rows, cols, ld, t, exps, planes, dld, pstride);
    else
      crt_split_rows_kernel<false, 32><<<grid, 256, 0, st>>>(A, rows, cols, ld, t, exps, planes, dld, pstride);
  }
  return cudaGetLastError();
}

long long round_up_ll(long long v, long long a) { return (v + a - 1) / a * a; }

// Split both operands, run the per-modulus slice GEMMs (residue bytes in Y,
// [nmod][M][ldy]) and, if out != NULL, reconstruct.  Y_user (optional) gets
// the residues as [nmod][M][N]; ea_user / eb_user the exponents.
df_status crt_gemm(const double *A, const double *B, int M, int N, int K, int nmod, double *out, uint8_t *Y_user,
                   int32_t *ea_user, int32_t *eb_user, cudaStream_t st) {
  if (!A || !B || M <= 0 || N <= 0 || K <= 0) return DF_ERR_ARG;
  CrtTab t;
  if (!make_tab(K, nmod, &t)) return DF_ERR_ARG;
  const long long ld = round_up_ll(K, 16);
  const long long ldy = round_up_ll(N, 16);
  // A B^T with B == A (a Gram matrix such as K_b = X_b X_b^T): one split serves both sides
  const bool same = A == B && M == N;
  uint16_t *Ad = nullptr, *Bd = nullptr;
  uint8_t *Y = nullptr;
  int *ea = nullptr, *eb = nullptr, *status = nullptr;
  df_status rs = DF_OK;
  cudaError_t e = scratch_malloc((void **)&Ad, sizeof(uint16_t) * (size_t)nmod * M * ld, st);
  if (e == cudaSuccess && !same) e = scratch_malloc((void **)&Bd, sizeof(uint16_t) * (size_t)nmod * N * ld, st);
  // partial residues and the upper tiles alone serve the reconstruction; the
  // inspection entry point returns whole products
  SgParams p;
  grid_params(&p, kModeMod, M, N, K, 1);  // shiftT[1] = 0: the sums are exact
  plan_mod_gemm(&p, nmod, same && out, out != nullptr);
  if (e == cudaSuccess) e = scratch_malloc((void **)&Y, (size_t)nmod * p.nsplit * M * ldy, st);
  if (e == cudaSuccess) e = scratch_malloc((void **)&ea, sizeof(int) * M, st);
  if (e == cudaSuccess && !same) e = scratch_malloc((void **)&eb, sizeof(int) * N, st);
  if (e == cudaSuccess) e = scratch_malloc((void **)&status, sizeof(int), st);
  if (e == cudaErrorMemoryAllocation) rs = DF_ERR_OOM;
  if (e == cudaSuccess) e = cudaMemsetAsync(status, 0, sizeof(int), st);
  if (e == cudaSuccess) e = launch_crt_split(A, M, K, K, t, ea, Ad, ld, (long long)M * ld, false, st);
  if (e == cudaSuccess && !same) e = launch_crt_split(B, N, K, K, t, eb, Bd, ld, (long long)N * ld, false, st);
  const uint16_t *Bplanes = same ? Ad : Bd;
  const int *ebx = same ? ea : eb;
  if (e == cudaSuccess) {
    SgMaps maps;
    const SgOperand a{Ad, K, M, nmod, ld, (long long)M * ld}, b{Bplanes, K, N, nmod, ld, (long long)N * ld};
    if (!make_operand_maps(&maps, a, b, kTile)) {
      rs = DF_ERR_CUDA;
    } else {
      p.out = reinterpret_cast<double *>(Y);
      p.out_ld = ldy;
      p.out_blk = (long long)M * ldy;
      p.status = status;
      for (int i = 0; i < nmod; ++i) p.crt_mod[i] = t.mod[i];
      if (p.shiftT[1] != 0 || (long long)p.nunits > (1ll << 30)) rs = DF_ERR_ARG;
      else e = launch_slice_gemm(p, maps, st);
    }
  }
  if (e == cudaSuccess && rs == DF_OK && out) {
    const long long plane = (long long)M * ldy;
    if (same) {
      static_assert(kModSplitMax == 4, "one reconstruction kernel per part count");
      auto kern = p.nsplit == 1   ? crt_reconstruct_sym_kernel<1>
                  : p.nsplit == 2 ? crt_reconstruct_sym_kernel<2>
                  : p.nsplit == 3 ? crt_reconstruct_sym_kernel<3>
                                  : crt_reconstruct_sym_kernel<4>;
      const unsigned nm = (unsigned)((N + 7) / 8);
      const dim3 grid((unsigned)((N + 31) / 32), nm < 65535 ? nm : 65535);
      kern<<<grid, 256, 0, st>>>(Y, N, ldy, plane, ea, t, out, N);
    } else {
      auto kern = p.nsplit == 1   ? crt_reconstruct_kernel<1>
                  : p.nsplit == 2 ? crt_reconstruct_kernel<2>
                  : p.nsplit == 3 ? crt_reconstruct_kernel<3>
                                  : crt_reconstruct_kernel<4>;
      const dim3 grid((unsigned)((N + 255) / 256), (unsigned)(M < 65535 ? M : 65535));
      kern<<<grid, 256, 0, st>>>(Y, M, N, ldy, plane, ea, ebx, t, out, N);
    }
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && rs == DF_OK && Y_user)
    e = cudaMemcpy2DAsync(Y_user, N, Y, ldy, N, (size_t)nmod * M, cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess && rs == DF_OK && ea_user)
    e = cudaMemcpyAsync(ea_user, ea, sizeof(int) * M, cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess && rs == DF_OK && eb_user)
    e = cudaMemcpyAsync(eb_user, ebx, sizeof(int) * N, cudaMemcpyDeviceToDevice, st);
  int h = 0;
  if (e == cudaSuccess && rs == DF_OK) e = cudaMemcpyAsync(&h, status, sizeof(int), cudaMemcpyDeviceToHost, st);
  for (void *ptr : {(void *)Ad, (void *)Bd, (void *)Y, (void *)ea, (void *)eb, (void *)status})
    if (ptr) cudaFreeAsync(ptr, st);
  const cudaError_t es = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = es;
  if (rs != DF_OK) return rs;
  if (e != cudaSuccess) return DF_ERR_CUDA;
  return h ? DF_ERR_TIMEOUT : DF_OK;
}

}  // namespace

}  // namespace df

extern "C" {

int df_crt_modulus(int i) {
  int mods[df::kCrtMaxModuli];
  if (i < 0 || i >= df::kCrtMaxModuli) return 0;
  df::greedy_moduli(df::kCrtMaxModuli, mods);
  return mods[i];
}

int df_crt_operand_bits(long long K, int nmod) { return df::operand_bits(K, nmod); }

int df_crt_moduli_for_bits(long long K, int bits) {
  for (int n = 2; n <= df::kCrtMaxModuli; ++n)
    if (df::operand_bits(K, n) >= bits + 1) return n;
  return 0;
}

df_status df_crt_split_rows(const double *A, int rows, int cols, int ld, int nmod, int32_t *exps, int16_t *res,
                            void *stream) {
  if (!A || !exps || !res || rows < 0 || cols <= 0 || ld < cols) return DF_ERR_ARG;
  df::CrtTab t;
  if (!df::make_tab(cols, nmod, &t)) return DF_ERR_ARG;
  const cudaError_t e = df::launch_crt_split(A, rows, cols, ld, t, exps, reinterpret_cast<uint16_t *>(res), cols,
                                             (long long)rows * cols, true, reinterpret_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? DF_OK : DF_ERR_CUDA;
}

df_status df_crt_residue_products(const double *A, const double *B, int M, int N, int K, int nmod, uint8_t *Y,
                                  int32_t *ea, int32_t *eb, void *stream) {
  if (!Y) return DF_ERR_ARG;
  return df::crt_gemm(A, B, M, N, K, nmod, nullptr, Y, ea, eb, reinterpret_cast<cudaStream_t>(stream));
}

df_status df_emulated_gemm_crt(const double *A, const double *B, int M, int N, int K, int nmod, double *out,
                               void *stream) {
  if (!out) return DF_ERR_ARG;
  return df::crt_gemm(A, B, M, N, K, nmod, out, nullptr, nullptr, nullptr, reinterpret_cast<cudaStream_t>(stream));
}

}  // extern "C"
