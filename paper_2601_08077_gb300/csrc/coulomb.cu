// Coulomb build in FP64 (Section 2.1, Eqs. df-j-1 and df-j-2) and the energy
// reductions.
//
//   rho_P = sum_mn B_Pmn D_mn     (one streaming pass over B)
//   J_mn  = sum_P B_Pmn rho_P     (a second streaming pass over B)
//
// Both B_P and D are symmetric (D by the paper's assumption in Section 2.1,
// B_P by construction), so each pass reads only the upper triangle of every
// B_P: nao(nao+1)/2 doubles per auxiliary function instead of nao^2.  That
// halves the DRAM bytes and the FP64 FMAs of the paper's 4 N_scr N_aux
// (Section 3.1).  On GB300 the FP64 pipe is narrow, so these kernels are
// bounded by FP64 FMA throughput rather than by HBM; the roofline reported
// for them uses the measured FP64 rate.
//
// B comes dense ([naux][nao][nao]) or packed (per P the upper triangle row by
// row, [naux][nao (nao + 1) / 2], the symmetric storage Section 3.3
// describes); both layouts are read in the same order, so rho and J are
// bit-identical between them.
//
// A Schwarz-screened B (Section 2.1: a screened AO pair is zero in every B_P)
// is block-sparse: with per-mu masks of the 64-wide nu chunks that hold a
// nonzero, both passes skip the zero chunks (rho loses only zero terms; J is
// exactly zero there), cutting bytes and FMAs to the surviving pairs.
#include "df_internal.h"

namespace df {

namespace {

// rho of G functions per CTA, whose 8 warps are the 8 parts: in row-pair order
// (G = 1, with offsets of type Off), or row by row for a B of mostly zero chunks.
template <bool kPacked, bool kRows, int G, int kCtas = 4, typename Off = int>
__global__ void __launch_bounds__(256, kCtas) rho_kernel(const double *__restrict__ B, const double *__restrict__ D,
                                                     int naux, int nao, const uint32_t *__restrict__ mask,
                                                     double *__restrict__ rho, double *__restrict__ rho2) {
  __shared__ double part[8][G];
  double v[G];
  const int P0 = blockIdx.x * G;
  if constexpr (kRows)
    rho_part_rows<kPacked, G>(B, D, naux, nao, mask, P0, threadIdx.x >> 5, v);
  else
    rho_part<kPacked, G, 8, Off>(B, D, naux, nao, P0, threadIdx.x >> 5, v);
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int g = 0; g < G; ++g) part[threadIdx.x >> 5][g] = v[g];
  __syncthreads();
  const int g = threadIdx.x;
  if (g < G && P0 + g < naux) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += part[w][g];
    rho[P0 + g] = t;
    if (rho2) rho2[P0 + g] = t;
  }
}

// J_mn = sum_P B_Pmn rho_P over the upper triangle, written to both halves.
// CTA (x, y) takes elements x*256 .. of the row pair (y, nao-1-y), so every CTA
// has the same work.  Each element's sum runs over P in ascending order, one FMA
// per P, with eight loads of B ahead of their FMAs.
template <bool kPacked>
__global__ void __launch_bounds__(256, 5) coulomb_kernel(const double *__restrict__ B,
                                                         const double *__restrict__ rho, int naux, int nao,
                                                         double *__restrict__ J,
                                                         const uint32_t *__restrict__ mask_mu) {
  extern __shared__ double srho[];
  for (int i = threadIdx.x; i < naux; i += blockDim.x) srho[i] = rho[i];
  __syncthreads();
  int mu, nu;
  if (!pair_element(nao, blockIdx.y, blockIdx.x * 256 + threadIdx.x, mu, nu)) return;
  double acc = 0.0;  // a screened pair: B_P mu nu = 0 for every P
  if (!mask_mu || ((__ldg(mask_mu + mu) >> (nu >> 6)) & 1u)) {
    const long long off = kPacked ? packed_row(mu, nao) + (nu - mu) : (long long)mu * nao + nu;
    const long long stride = kPacked ? (long long)nao * (nao + 1) / 2 : (long long)nao * nao;
    acc = coulomb_sum<8, false>(B + off, stride, srho, naux);
  }
  J[(long long)mu * nao + nu] = acc;
  J[(long long)nu * nao + mu] = acc;
}

// True in every thread of the last CTA of the grid to arrive here (each CTA's
// global writes before it are visible to that CTA).  The ticket wraps to zero at
// the last arrival in one atomic, so it is zero after any number of whole
// launches, also when two of them shared it at the same time.
__device__ __forceinline__ bool last_block(unsigned *ticket) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// Sum of the values of a 256-thread block, in thread 0 (fixed order).
__device__ __forceinline__ double block_sum(double v, double *red) {
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < 8; ++w) s += red[w];
  __syncthreads();
  return s;
}

// E[0] = 1/2 sum D.J, E[1] = 1/2 sum rho.rho, E[2] = -1/2 sum D.K: partial sums
// per block, added by the last block to finish (thread t takes blocks t, t + 256,
// ..., then the block sum: the same order on every run).  A second launch whose
// one thread walked 296 partials took 54 us of an SCF step of 204 (20 atoms).
__global__ void __launch_bounds__(256) energy_kernel(const double *__restrict__ D, const double *__restrict__ J,
                                                     const double *__restrict__ K, const double *__restrict__ rho,
                                                     long long n2, int naux, double *__restrict__ part,
                                                     unsigned *__restrict__ ticket, double *__restrict__ E) {
  double a = 0.0, b = 0.0, c = 0.0;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n2; i += stride) {
    const double d = D[i];
    if (J) a = fma(d, J[i], a);
    if (K) c = fma(d, K[i], c);
  }
  if (rho)
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < naux; i += stride)
      b = fma(rho[i], rho[i], b);
  __shared__ double red[8];
  a = block_sum(a, red);
  b = block_sum(b, red);
  c = block_sum(c, red);
  if (threadIdx.x == 0) {
    part[blockIdx.x * 3] = a;
    part[blockIdx.x * 3 + 1] = b;
    part[blockIdx.x * 3 + 2] = c;
  }
  if (!last_block(ticket)) return;
  a = b = c = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += 256) {
    a += __ldcg(part + 3 * i);
    b += __ldcg(part + 3 * i + 1);
    c += __ldcg(part + 3 * i + 2);
  }
  a = block_sum(a, red);
  b = block_sum(b, red);
  c = block_sum(c, red);
  if (threadIdx.x == 0) {
    E[0] = 0.5 * a;
    E[1] = 0.5 * b;
    E[2] = -0.5 * c;
  }
}

// *out = ||D - D_prev||_F (1 when there is no previous density), D_prev = D, in
// one pass; the last block adds the partial sums.
__global__ void __launch_bounds__(256) density_change_kernel(const double *__restrict__ D, double *__restrict__ Dprev,
                                                             bool have_prev, long long n2,
                                                             double *__restrict__ part,
                                                             unsigned *__restrict__ ticket,
                                                             double *__restrict__ out) {
  double a = 0.0;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n2; i += stride) {
    const double v = D[i];
    const double d = have_prev ? v - Dprev[i] : 0.0;
    Dprev[i] = v;
    a = fma(d, d, a);
  }
  __shared__ double red[8];
  a = block_sum(a, red);
  if (threadIdx.x == 0) part[blockIdx.x] = a;
  if (!last_block(ticket)) return;
  a = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += 256) a += __ldcg(part + i);
  a = block_sum(a, red);
  if (threadIdx.x == 0) *out = have_prev ? sqrt(a) : 1.0;
}

// Packed B: flag[k] = 1 when the packed pair k (of the upper triangle) is
// nonzero in some B_P (one coalesced pass over B), then the per-mu masks
// over all nu from the symmetric pair flags.
__global__ void __launch_bounds__(256) packed_pair_flags_kernel(const double *__restrict__ Bp, int naux,
                                                                long long npk, uint8_t *__restrict__ flag) {
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= npk) return;
  uint8_t f = 0;
  for (int P = 0; P < naux && !f; ++P) f = __ldg(Bp + (long long)P * npk + k) != 0.0;
  flag[k] = f;
}

__global__ void mask_from_packed_flags_kernel(const uint8_t *__restrict__ flag, int nao,
                                              uint32_t *__restrict__ mask_mu) {
  const int mu = blockIdx.x * blockDim.x + threadIdx.x;
  if (mu >= nao) return;
  uint32_t bits = 0u;
  for (int nu = 0; nu < nao; ++nu) {
    const long long k = nu >= mu ? packed_row(mu, nao) + (nu - mu) : packed_row(nu, nao) + (mu - nu);
    if (flag[k]) bits |= 1u << (nu >> 6);
  }
  mask_mu[mu] = bits;
}

// Dense copy of B_P for P = P0 .. P0 + nP - 1 from the packed layout.
__global__ void unpack_kernel(const double *__restrict__ Bp, int P0, int nP, int nao, double *__restrict__ out) {
  const long long npk = (long long)nao * (nao + 1) / 2;
  const long long n2 = (long long)nao * nao;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)nP * n2) return;
  const int pl = (int)(i / n2);
  const int mu = (int)((i - pl * n2) / nao), nu = (int)(i - pl * n2 - (long long)mu * nao);
  const int lo = mu < nu ? mu : nu, hi = mu < nu ? nu : mu;
  out[i] = __ldg(Bp + (long long)(P0 + pl) * npk + packed_row(lo, nao) + (hi - lo));
}

// Per 128-row tile t of the (P, mu) rows (row r has mu = r mod nao): the OR of
// its rows' masks.
__global__ void tile_mask_kernel(const uint32_t *__restrict__ mask_mu, int nao, long long rows, int ntiles,
                                 uint32_t *__restrict__ mask_tile) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ntiles) return;
  uint32_t m = 0u;
  const long long r0 = (long long)t * kTile;
  for (long long r = r0; r < r0 + kTile && r < rows; ++r) m |= mask_mu[r % nao];
  mask_tile[t] = m;
}

}  // namespace

constexpr int kEnergyBlocks = 296;

cudaError_t launch_pair_masks_packed(const double *Bp, int naux, int nao, uint32_t *mask_mu, cudaStream_t st) {
  const long long npk = (long long)nao * (nao + 1) / 2;
  uint8_t *flag = nullptr;
  cudaError_t e = cudaMallocAsync(reinterpret_cast<void **>(&flag), (size_t)npk, st);
  if (e != cudaSuccess) return e;
  packed_pair_flags_kernel<<<(unsigned)((npk + 255) / 256), 256, 0, st>>>(Bp, naux, npk, flag);
  e = cudaGetLastError();
  if (e == cudaSuccess) {
    mask_from_packed_flags_kernel<<<(nao + 127) / 128, 128, 0, st>>>(flag, nao, mask_mu);
    e = cudaGetLastError();
  }
  cudaFreeAsync(flag, st);
  return e;
}

cudaError_t launch_unpack(const double *Bp, int P0, int nP, int nao, double *out, cudaStream_t st) {
  const long long n = (long long)nP * nao * nao;
  unpack_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(Bp, P0, nP, nao, out);
  return cudaGetLastError();
}

cudaError_t launch_tile_masks(const uint32_t *mask_mu, int naux, int nao, uint32_t *mask_tile, cudaStream_t st) {
  const long long rows = (long long)naux * nao;
  const int ntiles = (int)((rows + kTile - 1) / kTile);
  tile_mask_kernel<<<(ntiles + 255) / 256, 256, 0, st>>>(mask_mu, nao, rows, ntiles, mask_tile);
  return cudaGetLastError();
}

cudaError_t launch_density_change(const double *D, double *Dprev, bool have_prev, long long n2, double *part,
                                  unsigned *ticket, double *out, cudaStream_t st) {
  density_change_kernel<<<kDensityChangeBlocks, 256, 0, st>>>(D, Dprev, have_prev, n2, part, ticket, out);
  return cudaGetLastError();
}

CoulombWork rho_work(const double *B, const double *D, int naux, int nao, bool packed, bool rows, const uint32_t *mask,
                     double *part, int *work) {
  CoulombWork w{};
  w.kind = 1;
  w.naux = naux;
  w.nao = nao;
  w.packed = packed;
  // 912 spare warps (6 on each of 152 SMs): as many functions at once (one load
  // of D serves the group) as leave every warp an item
  w.group = naux >= 456 && nao <= 16384 ? 4 : 1;
  w.nitems = 8 * ((naux + w.group - 1) / w.group);
  w.B = B;
  w.D = D;
  w.part = part;
  w.rows = rows;
  w.mask = mask;
  w.work = work;
  return w;
}

CoulombWork coulomb_work_of(const double *B, const double *rho, int naux, int nao, bool packed, const uint32_t *mask,
                            double *J, int *work) {
  CoulombWork w{};
  w.kind = 2;
  w.naux = naux;
  w.nao = nao;
  w.packed = packed;
  w.nitems = (nao + 1 + 31) / 32 * ((nao + 1) / 2);
  w.B = B;
  w.rho = rho;
  w.J = J;
  w.mask = mask;
  w.work = work;
  return w;
}

cudaError_t launch_rho(const double *B, const double *D, int naux, int nao, double *rho, double *rho2,
                       cudaStream_t st, const uint32_t *mask_mu, bool packed, bool rows, bool alone) {
  // row order: the walk over rows and masks costs more instructions than the FMAs,
  // so functions share it while the SMs keep two CTAs (350 AOs: 700 functions 130
  // us one by one, 102 by two, 113 by four; 1050 functions 145 by two, 114 by four)
  const int group = !rows ? 1 : naux >= 1024 ? 4 : naux >= 304 ? 2 : 1;
  // dense: a CTA a function, four of them an SM or, alone on the GPU, five if that takes less: a
  // wave of five is a quarter longer (152 SMs, 235 AOs and 705 functions: 60 us in two waves of
  // four, 51 in one of five; packed, 435 and 1305: 275 and 245; 600 and 1800, three waves of
  // either: 583 and 619).  A batch's rho and J run beside each other, where waves do not count (16
  // molecules' J and K 15.3 ms with fours, 15.6 with this rule).  At 48 registers 64-bit offsets
  // suit the dense layout (435 and 1305: 252 us for 300) and 32-bit ones the packed (254 for 270);
  // past 2^31 elements of a B_P they have to be 64-bit.
  const long long sms = slice_gemm_grid(1 << 30);
  const bool five = alone && (naux + 5 * sms - 1) / (5 * sms) * 5 < (naux + 4 * sms - 1) / (4 * sms) * 4;
  auto kern = packed ? rho_kernel<true, false, 1> : rho_kernel<false, false, 1>;
  if (five) kern = packed ? rho_kernel<true, false, 1, 5> : rho_kernel<false, false, 1, 5, long long>;
  if (nao > kRho32Nao) kern = packed ? rho_kernel<true, false, 1, 5, long long> : rho_kernel<false, false, 1, 5, long long>;
  if (rows && group == 4) kern = packed ? rho_kernel<true, true, 4> : rho_kernel<false, true, 4>;
  if (rows && group == 2) kern = packed ? rho_kernel<true, true, 2> : rho_kernel<false, true, 2>;
  if (rows && group == 1) kern = packed ? rho_kernel<true, true, 1> : rho_kernel<false, true, 1>;
  kern<<<(unsigned)((naux + group - 1) / group), 256, 0, st>>>(B, D, naux, nao, mask_mu, rho, rho2);
  return cudaGetLastError();
}

cudaError_t launch_coulomb(const double *B, const double *rho, int naux, int nao, double *J, cudaStream_t st,
                           const uint32_t *mask_mu, bool packed) {
  const size_t sm = (size_t)naux * sizeof(double);
  static size_t attr = 48 * 1024;
  if (sm > attr) {
    cudaError_t e = cudaFuncSetAttribute(coulomb_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(coulomb_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    attr = sm;
  }
  const dim3 g((nao + 1 + 255) / 256, (nao + 1) / 2);
  if (packed)
    coulomb_kernel<true><<<g, 256, sm, st>>>(B, rho, naux, nao, J, mask_mu);
  else
    coulomb_kernel<false><<<g, 256, sm, st>>>(B, rho, naux, nao, J, mask_mu);
  return cudaGetLastError();
}

cudaError_t launch_energy(const double *D, const double *J, const double *K, const double *rho, int nao, int naux,
                          double *partials, unsigned *ticket, double *E_dev, cudaStream_t st) {
  energy_kernel<<<kEnergyBlocks, 256, 0, st>>>(D, J, K, rho, (long long)nao * nao, naux, partials, ticket, E_dev);
  return cudaGetLastError();
}

}  // namespace df
