// Internal declarations of libdf: the context, the kernel launchers and the
// slice-GEMM work description.  Not part of the public ABI (include/df.h).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <cublas_v2.h>
#include <cstdint>
#include <vector>

#include "../../include/df.h"
#include "coulomb_dev.cuh"
#include "df_device.cuh"

namespace df {

constexpr int kTile = 128;       // output tile edge of the slice GEMM
constexpr int kKTile = 64;       // K elements per pipeline stage (128 bytes of bf16)
constexpr int kMaxChunk = 1024;  // products per exact FP32 accumulation chunk

// What a slice GEMM computes and how it stores it.
enum SgMode : int {
  kModeX = 0,       // first exchange GEMM, X = B C with the (P, mu) rows on the MMA's M side and the
                    // orbitals on its N side: the exact int64 sums R[m*ld + n] (the X split rounds them)
  kModeKPart = 1,   // second exchange GEMM: upper tile pairs of K_b = X_b X_b^T, an int64 fixed-point
                    // partial per (block, K split), raw[part*blk + n*ld + m] (the reduce scales and sums them)
  kModeRaw = 2,     // exact S_g per group: raw[(g*n_valid + n)*m_valid + m]
  kModeGemm = 3,    // generic emulated product: out[m*ld + n]
  kModeMod = 5,     // CRT variant: the exact sum of one modulus plane reduced modulo that
                    // modulus, one byte each: out8[plane*out_blk + m*ld + n]
};

constexpr int kCrtMaxModuli = 16;

// Blocks of the density-change reduction ||D - D_prev||_F (df_build_J).
constexpr int kDensityChangeBlocks = 152;

// Row splits give a whole 256-thread block to each row at least this wide
// (fewer, longer rows: the second exchange GEMM's operands), else a warp.
constexpr int kWideRow = 2048;

struct SgParams {
  int mode;
  int nunits;
  int nt_m, nt_n;           // tiles along m and n
  int m_valid, n_valid;     // rows of the A side and of the B side that exist
  int ktiles;               // K tiles (64 wide); kModeKPart: of a block, from nocc
  int kvalid;               // K values (the last tile's rest is zeros); kModeKPart: of a block, from nocc
  int nw;                   // columns of an n tile (rows of a stacked B digit): a multiple of 32, at most 128
  int q;                    // digits stacked in one MMA: min(8, 256 / nw)
  int s_fixed;              // slice count (kModeRaw, kModeGemm, kModeMod)
  int nao, nocc, nblk, naux;
  int nsplit;               // K splits per block (kModeKPart) or plane (kModeMod)
  int sym;                  // kModeMod: A == B, only the tiles (i, j >= i) are formed
  const int *s_blk;         // per-block slice counts (kModeX, kModeKPart)
  int shiftT[9];            // truncation T of the fixed-point sum, indexed by s (0..8)
  const int *ea;            // A-side row exponents
  const int *eb;            // B-side row exponents
  long long out_ld;
  long long out_blk;
  double *out;
  long long *raw;
  int *status;              // device status word (DF_ERR_TIMEOUT bits)
  // CTA-pair mode: two CTAs of a cluster take two tiles that share their
  // B-side operand; each CTA loads its own A tile and half of the stacked
  // B rows into its own shared memory (both copies complete on the first
  // CTA's barrier), and one M = 256 MMA reads both CTAs' tiles.  Work is
  // then counted in tile pairs (npairs); the host sets both.
  int pair;
  int npairs;
  int crt_mod[kCrtMaxModuli];  // kModeMod: the modulus of each plane
  // first exchange GEMM on a screened (block-sparse) B: per 128-row tile of
  // B's (P, mu) rows, the bit mask of its nonzero 64-wide K tiles (bit k = K
  // tile k, at most 32); null = dense
  const uint32_t *kmask;
  // first exchange GEMM (kModeX): per (block, mu) row of X, the
  // largest bit-length bound E = bitlen(|R|) + k over the row's nonzero exact
  // sums R (|R 2^k| < 2^E), atomically maxed; the X split takes it as its
  // exponent guess and so reads R once.  Reset to kRowBoundNone before the
  // launch; null = not recorded.
  int *rowE;
};

// "No nonzero element yet" in a row bound (the C split resets the bounds);
// below every real bound.
constexpr int kRowBoundNone = (int)0x80808080;

// Work units of a launch: tiles, and tile pairs in CTA-pair mode (0 = the
// mode has no pairing).
long long slice_gemm_units(const SgParams &p);
long long slice_gemm_pairs(const SgParams &p);

// One operand's digit planes: [planes][rows][ld] BF16, k of the ld columns used.
struct SgOperand {
  const void *base;
  long long k, rows, planes, ld, plane_stride;
};

// Tensor maps of a launch: boxes of 64 (K) x 128 rows of A, and of nw and
// nw / 2 rows of B (a CTA of a pair stages a digit's rows whole or by halves).
// x: the first exchange GEMM's output, for its TMA stores.
struct SgMaps {
  CUtensorMap a, b, h, x;
};
bool make_tmap_x(CUtensorMap *map, const void *base, long long ld, long long rows);
bool make_operand_maps(SgMaps *m, const SgOperand &a, const SgOperand &b, int nw);

// A stand-alone product of A [M][K] and B [N][K] over s digits (kModeRaw, kModeGemm):
// sizes, tiles and truncation; the caller sets the exponents and the output.
void grid_params(SgParams *p, int mode, int M, int N, int K, int s);

// CRT variant: the planes of a residue product, the upper tiles only (sym: A ==
// B, whose products are symmetric) and, if the caller can add partial residues,
// K splits, single tiles or CTA pairs: the fewest waves over the SMs or pairs of
// them, weighted with the cycles a K tile takes (515 a tile of its own, 370 a tile
// of a pair, which takes in 24 KB instead of 32) and 3000 for a unit's store.
// 600 rows, 240 K tiles, 12 moduli: 15 of 25 tiles, in pairs of two K parts, 105 us
// for 130.
constexpr int kModSplitMax = 4;
void plan_mod_gemm(SgParams *p, int planes, bool sym, bool split);

// A grouped launch: the work units of several problems (molecules) in one
// persistent launch.  Problem i owns units [unit_off[i], unit_off[i+1]); its
// parameters are params[i] and its tensor maps maps[4i] .. maps[4i+3]
// (an SgMaps), all in device memory (maps 64-byte aligned).
struct SgGroup {
  const SgParams *params;
  const CUtensorMap *maps;
  const int *unit_off;
  int nmol;
  int total;
};

struct Ctx;

// Scratch of the stand-alone emulated-GEMM entry points: stream-ordered
// allocations from the device's default pool, whose release threshold is
// raised once so that repeated calls reuse the memory instead of mapping it
// again (it stays reserved by the process until cudaDeviceReset).
inline cudaError_t scratch_malloc(void **p, size_t bytes, cudaStream_t st) {
  static bool kept[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 && !kept[dev]) {
    cudaMemPool_t pool;
    if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
      uint64_t thr = ~0ull;
      cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
    }
    kept[dev] = true;
  }
  return cudaMallocAsync(p, bytes, st);
}

// Kernel launchers (split.cu, slicegemm.cu, coulomb.cu).
cudaError_t launch_split_rows_bf16(const double *A, long long rows, int cols, long long ld, int nslices,
                                   int *exps, uint16_t *digits, long long dld, long long plane_stride,
                                   cudaStream_t st);
// Dense B [naux][nao][nao] at setup: *flag (zeroed first) set when some B_P is
// not exactly symmetric, the digits of its rows (P' = perm[P] order), and
// mask_mu (optional, nao <= 2048): per mu, bit c set when some B_P mu nu with
// nu in [64c, 64c + 64) is nonzero.
cudaError_t launch_setup_rows(const double *B, int naux, int nao, int nslices, int *exps, uint16_t *digits,
                              long long dld, long long plane_stride, const int *perm, uint32_t *mask_mu, int *flag,
                              cudaStream_t st);
cudaError_t launch_split_rows_int8(const double *A, int rows, int cols, int ld, int nslices, int *exps,
                                   int8_t *digits, cudaStream_t st);
// What the C split does on the way for the kernels after it: `reset` words set to
// kRowBoundNone, `zero` words set to 0.
struct ColsExtra {
  int *reset;
  int nreset;
  int *zero;
  int nzero;
};
cudaError_t launch_split_cols_bf16(const double *C, int nrows, int ncols, int nslices, int *exps,
                                   uint16_t *digits, long long dld, long long plane_stride, cudaStream_t st,
                                   const ColsExtra &extra);
struct ShiftTable {
  int v[9];
};
// R: the first GEMM's int64 sums (kModeX, nocc even: an odd count is padded
// with a zero orbital); X = fl64(R 2^k) is formed here with
// the first GEMM's exponents eB (rows (P, mu)), eC (orbitals), slices s_blk and
// truncation table T1, then split per (block, mu).  rowE: the first GEMM's
// per-row bound (SgParams::rowE).  rp: parts of rho to add on the way (part null: none).
cudaError_t launch_split_xblocks(const long long *R, int naux, int nao, int nocc, int nslices, const int *eB,
                                 const int *eC, const int *s_blk, const ShiftTable &T1, const int *rowE, int *eX,
                                 uint16_t *Xd, long long kb_ld, int nblk, const RhoParts &rp, cudaStream_t st);
cudaError_t launch_kpart_reduce(const long long *Rp, const int *eX, const int *s_blk, ShiftTable T, int nao,
                                int nblk, int nsplit, double *K, cudaStream_t st);

// Encode a 3D bf16 tensor map {k, rows, planes} with a 64 x box_rows x 1 box, 128B swizzle.
bool make_tmap_bf16(CUtensorMap *map, const void *base, long long k, long long rows, long long planes,
                    long long row_stride_elems, long long plane_stride_elems, int box_rows);

// cw (optional, the two exchange GEMMs): a Coulomb pass for the spare warps.
cudaError_t launch_slice_gemm(const SgParams &p, const SgMaps &m, cudaStream_t st, const CoulombWork *cw = nullptr);
// Grouped launch; `mode` is shared by all problems, `grid` CTAs (0 = one per SM).
// pairs: CTA-pair launch over tile pairs (kModeX only; unit_off and total
// count tile pairs, every problem's npairs set).
cudaError_t launch_slice_gemm_grouped(int mode, const SgGroup &g, int *status, int grid, cudaStream_t st,
                                      bool pairs = false);
int slice_gemm_grid(int nunits);
// One-thread kernel whose bounded wait on a never-completed mbarrier runs out
// after limit_ns and sets bit 0 of *status (bit 1: it returned without the
// abort path, which would be a defect).
cudaError_t launch_wait_selftest(int *status, unsigned long long limit_ns, cudaStream_t st);

// rho_P for every P into rho (and rho2 if given), J from rho.
// mask_mu (optional, block-sparse B): per mu, bit c set when some B_P mu nu
// with nu in [64c, 64c + 64) is nonzero; null = dense.
// packed: B holds per P the upper triangle row by row ([naux][nao (nao + 1) / 2]).
// rows: rho in the row-by-row order of a B of mostly zero chunks (nao <= 2048), else
// in row-pair order; the order is the B's, so a screened B gives the same bits
// with and without its masks.
// alone: no other launch is meant to run beside it.
cudaError_t launch_rho(const double *B, const double *D, int naux, int nao, double *rho, double *rho2,
                       cudaStream_t st, const uint32_t *mask_mu, bool packed, bool rows, bool alone);
cudaError_t launch_coulomb(const double *B, const double *rho, int naux, int nao, double *J, cudaStream_t st,
                           const uint32_t *mask_mu, bool packed);
// The same passes as work for a slice GEMM's spare warps: `work` is zeroed before
// the launch, part holds 8 naux doubles.
CoulombWork rho_work(const double *B, const double *D, int naux, int nao, bool packed, bool rows, const uint32_t *mask,
                     double *part, int *work);
CoulombWork coulomb_work_of(const double *B, const double *rho, int naux, int nao, bool packed, const uint32_t *mask,
                            double *J, int *work);
// The masks of a packed B (pair flags through stream-ordered scratch of nao (nao + 1) / 2 bytes).
cudaError_t launch_pair_masks_packed(const double *Bp, int naux, int nao, uint32_t *mask_mu, cudaStream_t st);
// Dense B_P, P = P0 .. P0 + nP - 1, into out [nP][nao][nao] from a packed B.
cudaError_t launch_unpack(const double *Bp, int P0, int nP, int nao, double *out, cudaStream_t st);
// Digits of B from its packed layout (rows (P', mu) as launch_split_rows_bf16 writes them).
cudaError_t launch_split_rows_packed(const double *Bp, int naux, int nao, int nslices, int *exps, uint16_t *digits,
                                     long long dld, long long plane_stride, const int *perm, cudaStream_t st);
// Per 128-row tile of the (P, mu) rows, the OR of its rows' mu masks.
cudaError_t launch_tile_masks(const uint32_t *mask_mu, int naux, int nao, uint32_t *mask_tile, cudaStream_t st);
cudaError_t launch_energy(const double *D, const double *J, const double *K, const double *rho, int nao,
                          int naux, double *partials, unsigned *ticket, double *E_dev, cudaStream_t st);

}  // namespace df
