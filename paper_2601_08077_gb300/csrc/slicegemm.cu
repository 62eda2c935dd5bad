// Slice GEMM on the 5th-generation tensor cores (tcgen05 + TMEM + TMA).
//
// Computes, for an output tile of 128 (A-side rows) x up to 128 (B-side rows),
// the exact slice-pair sums of Section 3.2
//
//     S_g = sum_{t+u=g} A_t B_u^T,   g = 0 .. s-1,
//
// where A_t, B_u are INT8 digit planes (row-major, K contiguous), and folds
// them into the fixed-point value R = sum_g 2^(8(s-1-g)) S_g, which the
// epilogue stores as it is or turns into FP64 with the power-of-two scales.
//
// GB300 mapping.  ptxas rejects tcgen05 .kind::i8 on sm_103a, so the digits
// are stored as BF16 (every integer in [-256, 256] is exact in BF16) and run
// through tcgen05.mma .kind::f16 with FP32 accumulators in TMEM.  A product of
// two digits is at most 2^14 in magnitude, so an accumulation of at most 1024
// products stays within 2^24 and is exact in FP32; an accumulator is therefore
// drained after at most 1024 products: the epilogue warps add it, converted to
// integers and shifted by its group's weight, into an int64 fixed-point total
// held in registers (64 per thread).
//
// Order of work.  A digit's tile has nw columns (128, or less where the B side
// has fewer rows: the first exchange GEMM cuts its orbitals into tiles of a
// multiple of 32), and q = min(8, 256 / nw) digits are stacked in one MMA's N
// side (N <= 256).  The groups are taken q at a time
// ("passes" g = glo .. ghi); group glo + j accumulates in columns
// j nw .. (j+1) nw of one 256-column TMEM buffer (two buffers: the tensor core
// fills one while the epilogue drains the other).  Step t of a pass multiplies
// A_t with the stacked B_{max(0, glo-t)} .. B_{ghi-t}: every issued column
// belongs to a slice pair of the triangle, so s(s+1)/2 pairs cost exactly
// s(s+1)/2 nw columns.  (Measured on GB300 with operands resident: an M = 128
// or cta_group::2 M = 256 MMA takes N / 2 cycles down to N = 128, 46-48 at
// N = 64; the stacking in fixed pairs that this replaced padded every odd row
// of the triangle to N = 256.)  The K range is cut into chunks of at most 16
// stages; all passes run on a chunk before the next one, so its digit tiles
// are re-read from L2.  Where a chunk is short, up to 16 / (its length)
// consecutive steps of a pass share their accumulators (at most 1024 products
// still), which saves drains: at 5 K tiles and 5 slices, 7 drained tiles for 15.
//
// Warp roles (384 threads, one CTA per SM, persistent over work units):
//   warp 0      TMA producer: 64-wide BF16 boxes of A_t and the stacked B
//               digits, 128B swizzle, into a ring guarded by mbarriers;
//   warp 1      TMEM allocation and the single-thread tcgen05.mma issuer;
//   warps 2, 3  idle (they give their registers to the epilogue: setmaxnreg), or, in the
//               512-thread form with warps 12 to 15, a Coulomb pass (kHelp, below);
//   warps 4..11 epilogue; warp w reads TMEM lanes 32*(w%4)..+31 (tile rows)
//               and half (w-4)/4 of each digit's columns.
// The producer's and the issuer's loops bound the kernel when they are written
// as one thread's code: measured with operands resident, a stage of four MMAs
// took 551 cycles to issue (a barrier wait ~175-210 of them even when the phase
// is complete), against 256 (N = 128) or 512 (N = 256) cycles of tensor work.
// So the whole warp runs each loop with warp-uniform control flow and an
// elected lane issues (operands in uniform registers), the next stage's barrier
// is polled (test_wait) before the current stage's work is issued, and the ring
// position and phases live in registers: 302 cycles per stage at N = 128.
//
// CTA-pair mode (cluster of two): rank 0's MMA issuer runs tcgen05.mma
// .cta_group::2 with M = 256 over two output tiles that share the B operand;
// each CTA stages its own A tile and half of the stacked B rows (a 6-stage
// ring of 32 KB), both CTAs' copies complete on rank 0's barriers, the commits
// arrive on both CTAs' barriers, and each CTA drains its own TMEM.
//
// Every mbarrier wait is bounded (4 s of wall clock); a wait that runs out
// sets a shared abort flag and bit 1 of the device status word, every role
// leaves its loop, the producer waits (bounded) for its copies in flight, the
// MMA issuer waits (bounded) for its MMAs, and the TMEM is freed.
#include "df_internal.h"

#include <climits>
#include <cstdio>
#include <cstring>
#include <type_traits>

namespace df {

namespace {

constexpr int kStages = 4;
constexpr int kTileBytes = kTile * kKTile * 2;        // one 128 x 64 BF16 box, 16 KB
constexpr int kStageBytes = 3 * kTileBytes;           // A_t tile + up to 256 stacked B rows
// CTA-pair mode (cta_group::2): a CTA stages its own A_t tile and half of the
// stacked B rows, so a stage is 32 KB and six fit in the space of the four
// 48 KB stages (seven measured no faster on GB300).
constexpr int kStagesP = 6;
constexpr int kStageBytesP = 2 * kTileBytes;
constexpr int kThreads = 384;                         // 12 warps
constexpr int kThreadsHelp = 512;                     // and 4 more spare warps for a Coulomb pass
constexpr int kEpiWarp0 = 4;
constexpr int kEpiWarps = 8;
constexpr int kAccBufs = 2;
constexpr uint32_t kAccCols = 256;                    // one accumulator buffer: the stacked digits' columns
constexpr uint32_t kTmemCols = 512;
constexpr int kChunkStages = kMaxChunk / kKTile;      // 16 stages = 1024 products
constexpr int kChunkX = 5;                            // K tiles per chunk of the first exchange GEMM
constexpr uint64_t kTimeoutNs = 4000000000ull;
constexpr int kBarBytes = 1024;
// Row-major stores go through shared memory, 8 columns of a warp's 32 rows at a
// time.  First exchange GEMM: two 2 KB patches per warp in the 64-byte swizzle
// that its TMA stores read.  Stand-alone product: 80 bytes per row (16-byte
// accesses by 8 lanes hit all 32 banks).
constexpr int kStoreCols = 8;
constexpr int kTmaPatch = 32 * kStoreCols * 8;
constexpr int kPatchPitch = 80;
constexpr int kPatchBytes = 2 * kTmaPatch;
static_assert(kPatchBytes >= 32 * kPatchPitch, "one patch serves both kinds of store");
constexpr int kSlack = 1024;                          // alignment of the ring
// CRT variant (kModeMod): one B tile per stage and short units (one plane,
// K / 64 stages each) streaming a large A operand, so the ring is deepened
// to keep more DRAM reads in flight.
constexpr int kStagesM = 7;
__host__ __device__ constexpr int ring_stages(int mode, bool pair) {
  return pair ? kStagesP : mode == kModeMod ? kStagesM : kStages;
}
__host__ __device__ constexpr int stage_bytes(int mode, bool pair) {
  return pair || mode == kModeMod ? kStageBytesP : kStageBytes;
}
__host__ __device__ constexpr int ring_bytes(int mode, bool pair) {
  return ring_stages(mode, pair) * stage_bytes(mode, pair);
}
constexpr bool mode_patch(int mode) { return mode == kModeX || mode == kModeGemm; }
constexpr int smem_bytes(int mode, bool pair) {
  return ring_bytes(mode, pair) + kBarBytes + (mode_patch(mode) ? kEpiWarps * kPatchBytes : 0) + kSlack;
}
static_assert(smem_bytes(kModeX, true) <= 232448 && smem_bytes(kModeX, false) <= 232448 &&
                  smem_bytes(kModeMod, false) <= 232448,
              "the ring must fit the 227 KB opt-in shared memory of a CTA");
// Register split (setmaxnreg): warps 0-3 drop to 64, the 8 epilogue warps rise
// to 216; 128*64 + 256*216 = 63488 <= 384 threads * 168 registers at launch.
constexpr int kRegsLow = 64;
constexpr int kRegsHigh = 216;
static_assert(128 * kRegsLow + 256 * kRegsHigh <= kThreads * 168, "register split exceeds the launch's registers");
// With the Coulomb warps: 256*56 + 256*200 = 65536 = 512 threads * 128 registers.
constexpr int kRegsLowH = 56;
constexpr int kRegsHighH = 200;
static_assert(256 * kRegsLowH + 256 * kRegsHighH <= kThreadsHelp * 128, "register split exceeds the launch's registers");

// Instruction descriptor of tcgen05.mma .kind::f16, BF16 x BF16 -> FP32, both
// operands K-major (D fmt bits 4-5, A fmt 7-9, B fmt 10-12, N>>3 at 17-22,
// M>>4 at 24-28); N is added at run time.  M = 128, or 256 across a CTA pair
// (128 rows of A in each CTA, the first half of the B rows in the first
// CTA's shared memory, the second half in the second's).
constexpr uint32_t idesc_base(int m) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(m >> 4) << 24);
}
constexpr uint32_t kIdesc1 = idesc_base(128);
constexpr uint32_t kIdesc2 = idesc_base(256);
__device__ __forceinline__ uint32_t idesc_n(uint32_t base, int n) { return base | ((uint32_t)(n >> 3) << 17); }

struct Unit {
  int m0, n0, m_end, az0, azs, bz0, bzs, kt0, ktiles, s, blk, part;
  int ksteps_last;  // 16-wide K steps of the unit's last K tile (the rest of that tile is zeros)
  // block-sparse K (first exchange GEMM on a screened B): the unit's nonzero
  // K tiles as a bit mask; ktiles then counts its set bits
  int sparse;
  uint32_t kmask;
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Acquire at cluster scope: the barrier may complete through arrivals or
// copies issued by the other CTA of a pair.
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Non-blocking poll of a barrier's phase.
template <bool kCluster>
__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  if (kCluster)
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
  return ok != 0;
}

// Bounded wait.  Returns false if the CTA is aborting or the wait ran out.
template <bool kCluster = false>
__device__ __forceinline__ bool wait_bounded(uint64_t *bar, uint32_t parity, volatile int *abort_flag,
                                             int *status, bool honour_abort = true,
                                             uint64_t limit_ns = kTimeoutNs) {
  auto poll = [&]() { return kCluster ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity); };
  if (poll()) return true;
  const uint64_t t0 = globaltimer_ns();
  while (true) {
    if (poll()) return true;
    if (honour_abort && *abort_flag) return false;
    if (globaltimer_ns() - t0 > limit_ns) {
      *abort_flag = 1;
      atomicOr(status, 1);
      return false;
    }
  }
}

__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1,
                                            int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
      : "memory");
}

// TMA store of a box of this CTA's shared memory (issued and committed by one thread).
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, const void *src, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(smem_u32(src)), "r"(c0), "r"(c1)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// The issuing thread: until all but one of its stores have read their shared memory / all are done.
__device__ __forceinline__ void tma_store_wait_read1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row core
// groups 1024 bytes apart (SBO), descriptor version 1, swizzle mode 2.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void umma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}

// --- CTA pair (cta_group::2) ---------------------------------------------
// TMA load into this CTA's shared memory that completes its bytes on the
// mbarrier at shared::cluster address `mbar` (rank 0's, for both CTAs).
__device__ __forceinline__ void tma_load_3d_pair(void *dst, const CUtensorMap *map, uint32_t mbar, int c0, int c1,
                                                 int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(mbar)
      : "memory");
}

// One thread of the first CTA issues the M = 256 MMA for both CTAs.
__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                               uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Arrive (once the pair's MMAs issued so far are done) on the barrier at the
// same offset in both CTAs of the pair.
__device__ __forceinline__ void umma_commit_pair(uint64_t *bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}

// Shared::cluster address of this CTA's variable `p` in CTA `rank`.
__device__ __forceinline__ uint32_t peer_addr(const void *p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
  return r;
}

// Arrive on a barrier of either CTA of the pair.  Default semantics: what the
// arrival publishes (TMEM reads done) is ordered by the tcgen05 fences around
// it, so no cluster-scope release (a full memory barrier) is needed.
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

// Every thread of both CTAs of the cluster.
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// One lane of a converged warp, known to the compiler as such: what runs under
// it (copies, MMAs) then takes its operands from uniform registers.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(p));
  return p != 0;
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// 32 (or 16, into the first half) consecutive TMEM columns of the thread's lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15])
      : "r"(taddr));
}

// Waits for the warp's TMEM loads; the registers are operands of volatile
// statements, so that nothing that uses them can be scheduled before the wait.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&a)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; i += 8)
    asm volatile(""
                 : "+r"(a[i]), "+r"(a[i + 1]), "+r"(a[i + 2]), "+r"(a[i + 3]), "+r"(a[i + 4]), "+r"(a[i + 5]),
                   "+r"(a[i + 6]), "+r"(a[i + 7])
                 :
                 : "memory");
}

// 16-wide K steps of the last K tile of a range of kvalid values.
__device__ __forceinline__ int tail_steps(int kvalid) {
  const int rem = (kvalid - 1) % kKTile + 1;
  return (rem + 15) >> 4;
}

// Tile (i, j) of block-and-split index bs of the second exchange GEMM.
__device__ __forceinline__ Unit kpart_unit(const SgParams &p, int i, int j, int bs) {
  Unit w;
  const int b = bs / p.nsplit;
  const int sp = bs - b * p.nsplit;
  w.m0 = i * kTile;
  w.n0 = j * kTile;
  w.m_end = p.m_valid;
  w.az0 = b;
  w.azs = p.nblk;
  w.bz0 = b;
  w.bzs = p.nblk;
  const int nP = min(kBlock, p.naux - b * kBlock);
  const int kt_b = (nP * p.nocc + kKTile - 1) / kKTile;
  w.kt0 = (int)((long long)kt_b * sp / p.nsplit);
  w.ktiles = (int)((long long)kt_b * (sp + 1) / p.nsplit) - w.kt0;
  w.ksteps_last = sp + 1 == p.nsplit ? tail_steps(nP * p.nocc) : kKTile / 16;
  w.s = p.s_blk[b];
  w.blk = b;
  w.part = bs;
  w.sparse = 0;
  w.kmask = 0u;
  return w;
}

// Tile (mt, nt) of a stand-alone product (kModeRaw, kModeGemm, kModeMod).
__device__ __forceinline__ Unit grid_unit(const SgParams &p, int mt, int nt) {
  Unit w;
  w.m0 = mt * kTile;
  w.n0 = nt * kTile;
  w.m_end = p.m_valid;
  w.az0 = 0;
  w.azs = 1;
  w.bz0 = 0;
  w.bzs = 1;
  w.kt0 = 0;
  w.part = 0;
  w.ktiles = p.ktiles;
  w.ksteps_last = tail_steps(p.kvalid);
  w.sparse = 0;
  w.kmask = 0u;
  w.blk = 0;
  w.s = p.s_fixed;
  return w;
}

// First exchange GEMM: unit u is an orbital tile (the inner index, so the B
// digits of a row tile are re-read from L2) of a row tile.  A row tile is 128
// (P, mu) rows, or 256 over a CTA pair, of ONE auxiliary block (128 nao rows):
// the last tile of a block may overhang its end (rows past m_end are computed
// and dropped), so both CTAs of a pair run the block's slice count whatever
// the parity of nao.
template <bool kPair>
__device__ __forceinline__ Unit x_unit(const SgParams &p, int u, int rank) {
  Unit w;
  constexpr int rows = kPair ? 2 * kTile : kTile;
  const int mt = u / p.nt_n, nt = u - mt * p.nt_n;
  const int per_block = (kBlock * p.nao + rows - 1) / rows;
  w.blk = mt / per_block;
  const int b0 = w.blk * kBlock * p.nao;
  const int base = b0 + (mt - w.blk * per_block) * rows;
  w.m0 = base + (kPair ? rank * kTile : 0);
  w.m_end = min(p.m_valid, b0 + kBlock * p.nao);
  w.n0 = nt * p.nw;
  w.az0 = 0;
  w.azs = 1;
  w.bz0 = 0;
  w.bzs = 1;
  w.kt0 = 0;
  w.part = 0;
  w.ktiles = p.ktiles;
  w.ksteps_last = tail_steps(p.kvalid);
  w.sparse = 0;
  w.kmask = 0u;
  w.s = p.s_blk[w.blk];
  if (p.kmask) {
    // block-sparse: the nonzero K tiles; a pair runs the union of its two tiles' (one MMA covers both)
    w.sparse = 1;
    w.kmask = p.kmask[base / kTile];
    if (kPair && base + kTile < w.m_end) w.kmask |= p.kmask[base / kTile + 1];
    w.ktiles = __popc(w.kmask);
    w.ksteps_last = kKTile / 16;
  }
  return w;
}

// Unit u of CTA `rank` of a pair (0 without pairs).  In the second exchange
// GEMM the pairs of (block, split) bs are the tiles (2a + r, j), j = 2a ..
// nt-1: the pair at j = 2a also computes the lower tile (2a+1, 2a), whose
// values are the transpose of an upper tile and are never read, and an m tile
// past the last one reads zeros and stores nothing.
template <int kMode, bool kPair>
__device__ __forceinline__ Unit decode_unit(const SgParams &p, int u, int rank) {
  if constexpr (kMode == kModeX) {
    return x_unit<kPair>(p, u, rank);
  } else if constexpr (kMode == kModeKPart) {
    // u -> (block b, K split sp, upper tile pair); block-major for L2 reuse
    const int nt = p.nt_m;
    if (kPair) {
      const int na = (nt + 1) / 2;
      const int per = na * (nt - na + 1);  // sum over a < na of (nt - 2a)
      const int pr = u % per;
      int a = 0, rem = pr;
      while (rem >= nt - 2 * a) {
        rem -= nt - 2 * a;
        ++a;
      }
      return kpart_unit(p, 2 * a + rank, 2 * a + rem, u / per);
    }
    const int npairs = nt * (nt + 1) / 2;
    const int pr = u % npairs;
    int i = 0, rem = pr;
    while (rem >= nt - i) {
      rem -= nt - i;
      ++i;
    }
    return kpart_unit(p, i, i + rem, u / npairs);
  } else if constexpr (kMode == kModeMod) {
    // plane- and K-split-major, so the tiles of a plane's K range are reused from L2
    const int na = kPair ? (p.nt_m + 1) / 2 : p.nt_m;
    const int per = p.sym ? (kPair ? na * (p.nt_m - na + 1) : na * (na + 1) / 2) : na * p.nt_n;
    const int ps = u / per, r = u % per;
    int i, j;
    if (p.sym) {
      i = 0;
      int rem = r;
      while (rem >= p.nt_m - (kPair ? 2 * i : i)) {
        rem -= p.nt_m - (kPair ? 2 * i : i);
        ++i;
      }
      if (kPair) i = 2 * i;
      j = i + rem;
      i += rank;
    } else {
      i = kPair ? 2 * (r % na) + rank : r % na;
      j = r / na;
    }
    Unit w = grid_unit(p, i, j);
    const int plane = ps / p.nsplit, sp = ps - plane * p.nsplit;
    w.az0 = plane;
    w.bz0 = plane;
    w.blk = plane;
    w.part = ps;
    w.kt0 = p.ktiles * sp / p.nsplit;
    w.ktiles = p.ktiles * (sp + 1) / p.nsplit - w.kt0;
    if (sp + 1 < p.nsplit) w.ksteps_last = kKTile / 16;
    return w;
  } else {
    if (kPair) {
      const int na = (p.nt_m + 1) / 2;
      return grid_unit(p, 2 * (u % na) + rank, u / na);
    }
    return grid_unit(p, u % p.nt_m, u / p.nt_m);
  }
}

// v mod m for 0 <= v < 2^32 and 2 <= m <= 256 with magic = ceil(2^32 / m):
// the high word of v * magic is floor(v / m) or one more, so one correction.
__device__ __forceinline__ int umod_barrett(uint32_t v, int m, uint32_t magic) {
  const int r = (int)(v - __umulhi(v, magic) * (uint32_t)m);
  return r < 0 ? r + m : r;
}

// R mod m in [0, m) for |R| < 2^40: R = a 2^24 + b with |a| < 2^16 and
// 0 <= b < 2^24; a 2^24 = a c24 (mod m) with c24 = 2^24 mod m, |a c24| < 2^24,
// made non-negative by off24, a multiple of m >= 2^24.
__device__ __forceinline__ int mod_i40(long long R, int m, uint32_t magic, int c24, int off24) {
  const int a = (int)(R >> 24);
  const uint32_t b = (uint32_t)(R & 0xFFFFFF);
  const int r = umod_barrett((uint32_t)(a * c24 + off24), m, magic) + umod_barrett(b, m, magic);
  return r >= m ? r - m : r;
}

__device__ __forceinline__ int bit_length(long long r) {
  const uint64_t u = r < 0 ? (uint64_t)(-(r + 1)) + 1ull : (uint64_t)r;
  const uint32_t hi = (uint32_t)(u >> 32);
  return (hi ? 64 : 32) - __clz((int)(hi ? hi : (uint32_t)u));
}

// The exponents of the thread's hw columns in the warp's patch (64 ints, 0 past n_valid).
// Returns the largest of them (INT_MIN if there is none).
__device__ __forceinline__ int stage_column_exponents(uint8_t *patch, const int *eb, int n0c, int n_valid, int hw,
                                                      int lane) {
  int *e = reinterpret_cast<int *>(patch);
  int emax = INT_MIN;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int j = 32 * h + lane;
    const bool valid = j < hw && n0c + j < n_valid;
    const int v = valid ? __ldg(eb + n0c + j) : 0;
    e[j] = v;
    if (valid) emax = max(emax, v);
  }
  emax = __reduce_max_sync(0xffffffffu, emax);
  __syncwarp();
  return emax;
}

// First exchange GEMM: this unit's part of the per-(block, mu) bound on the
// exponent of each X row (SgParams::rowE).  An element's exact sum R with
// exponent sum k has |R 2^k| < 2^E, E = bitlen(|R|) + k; the row bound is the
// largest E of its nonzero elements.  The thread's row is one (P, mu), its
// columns orbitals (columns past n_valid have R = 0), their exponents staged in
// the patch.  bitlen(x | y) is the larger bit length, so the elements, shifted
// to the largest column exponent emax and to a 31-bit window whose top is the
// sums' bound 2^wtop, are or-ed and one bit length is taken: 5 instructions an
// element (a bit length each took 15).  A row that vanishes in the window takes
// them one by one.  |R| - 1 stands for |R| of a negative R: one bit less for an
// exact power of two, a bound one too low, which the X split detects.
__device__ __forceinline__ void record_row_bound(const SgParams &p, const Unit &w, int m, int hw, int wtop,
                                                 const long long (&R)[64], int kexp_base, const uint8_t *patch,
                                                 int emax) {
  if (m >= w.m_end) return;
  const int sb = max(0, wtop - 31);
  uint32_t any = 0u;
#pragma unroll
  for (int j4 = 0; j4 < 16; ++j4) {
    if (4 * j4 >= hw) break;
    const int4 e = reinterpret_cast<const int4 *>(patch)[j4];
    const int ee[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int v = (int)(R[4 * j4 + i] >> sb);
      any |= (uint32_t)(v ^ (v >> 31)) >> min(emax - ee[i], 31);
    }
  }
  int best = kRowBoundNone;
  if (any) {
    best = 32 - __clz((int)any) + sb + emax;
  } else {
#pragma unroll 1
    for (int j4 = 0; 4 * j4 < hw; ++j4) {
      const int4 e = reinterpret_cast<const int4 *>(patch)[j4];
      const int ee[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        long long r = 0;
#pragma unroll
        for (int j = 0; j < 64; j += 4) r = j == 4 * j4 ? R[j + i] : r;
        if (r != 0) best = max(best, bit_length(r) + ee[i]);
      }
    }
  }
  if (best != kRowBoundNone) atomicMax(p.rowE + w.blk * p.nao + m % p.nao, best + kexp_base + __ldg(p.ea + m));
}

// Store of a warp's 32 rows x hw columns of X's sums by TMA, from two patches
// in turn: the warp's writes go out asynchronously, in 64-byte pieces of a row.
// 32 rows starting at a multiple of 32 never straddle an auxiliary block's end
// (128 nao rows); the tensor map clips the rows and columns past X's end.
__device__ __forceinline__ void store_x(uint8_t *patch, const CUtensorMap *map, int row0, int row_end, int n0c,
                                        int n_valid, int hw, const long long (&R)[64], int lane) {
  if (row0 >= row_end) return;  // the whole warp
#pragma unroll
  for (int c8 = 0; c8 < 8; ++c8) {
    const int nc = n0c + kStoreCols * c8;
    if (kStoreCols * c8 >= hw || nc >= n_valid) break;
    uint8_t *mine = patch + (c8 & 1) * kTmaPatch + lane * (kStoreCols * 8);
    if (lane == 0) tma_store_wait_read1();
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 4; ++j)
      *reinterpret_cast<ulonglong2 *>(mine + ((j ^ ((lane >> 1) & 3)) << 4)) =
          make_ulonglong2((unsigned long long)R[8 * c8 + 2 * j], (unsigned long long)R[8 * c8 + 2 * j + 1]);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (lane == 0) tma_store_2d(map, patch + (c8 & 1) * kTmaPatch, nc, row0);
  }
}

// Row-major store of a warp's 32 rows x hw columns (64-bit values), through
// the warp's shared-memory patch: a thread holds a row, and 32 rows written
// straight from the registers touch 32 lines per instruction; from the patch
// a warp writes whole 64-byte pieces of 8 rows.  16-byte accesses when the
// rows are 16-byte aligned (even ld, even first column).
__device__ __forceinline__ void store_rows(uint8_t *patch, unsigned long long *out, long long ld, int row0, int row_end,
                                           int n0c, int n_valid, int hw, const long long (&R)[64], int lane) {
  const bool wide = ((ld & 1) == 0) && ((n0c & 1) == 0) && ((reinterpret_cast<uintptr_t>(out) & 15) == 0);
#pragma unroll
  for (int c8 = 0; c8 < 8; ++c8) {
    if (8 * c8 >= hw) break;
    const int nc = n0c + 8 * c8;
    if (nc >= n_valid) break;
    ulonglong2 *mine = reinterpret_cast<ulonglong2 *>(patch + lane * kPatchPitch);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      mine[j] = make_ulonglong2((unsigned long long)R[8 * c8 + 2 * j], (unsigned long long)R[8 * c8 + 2 * j + 1]);
    __syncwarp();
    if (wide) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = 8 * i + (lane >> 2), c = 2 * (lane & 3);
        const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(patch + r * kPatchPitch + 8 * c);
        const int m = row0 + r, n = nc + c;
        if (m < row_end && n + 1 < n_valid)
          *reinterpret_cast<ulonglong2 *>(out + (long long)m * ld + n) = v;
        else if (m < row_end && n < n_valid)
          out[(long long)m * ld + n] = v.x;
      }
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int r = 4 * i + (lane >> 3), c = lane & 7;
        const unsigned long long v = *reinterpret_cast<const unsigned long long *>(patch + r * kPatchPitch + 8 * c);
        const int m = row0 + r, n = nc + c;
        if (m < row_end && n < n_valid) out[(long long)m * ld + n] = v;
      }
    }
    __syncwarp();
  }
}

// Epilogue store of the thread's columns n0c .. n0c + hw - 1 of row m (row0: the warp's first row).
template <int kMode>
__device__ __forceinline__ void store_tile(const SgParams &p, const Unit &w, int m, int row0, int n0c, int hw,
                                           long long (&R)[64], int kexp_base, uint8_t *patch, int lane) {
  if constexpr (kMode == kModeMod) {
    // CRT variant: y = S mod m_plane, one byte per element, row-major per plane
    if (m >= p.m_valid) return;
    const int md = p.crt_mod[w.blk];
    const uint32_t magic = 0xFFFFFFFFu / (uint32_t)md + 1u;
    const int c24 = (int)((1u << 24) % (unsigned)md);
    const int off24 = (int)(((1u << 24) + (unsigned)md - 1u) / (unsigned)md * (unsigned)md);
    uint8_t *out = reinterpret_cast<uint8_t *>(p.out) + (long long)w.part * p.out_blk + (long long)m * p.out_ld + n0c;
    if (n0c + 64 <= p.n_valid) {
#pragma unroll
      for (int j8 = 0; j8 < 8; ++j8) {
        uint64_t word = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) word |= (uint64_t)mod_i40(R[8 * j8 + j], md, magic, c24, off24) << (8 * j);
        reinterpret_cast<uint64_t *>(out)[j8] = word;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 64; ++j)
        if (n0c + j < p.n_valid) out[j] = (uint8_t)mod_i40(R[j], md, magic, c24, off24);
    }
  } else if constexpr (kMode == kModeGemm) {
    const int km = kexp_base + (m < p.m_valid ? __ldg(p.ea + m) : 0);
    stage_column_exponents(patch, p.eb, n0c, p.n_valid, hw, lane);
#pragma unroll
    for (int j4 = 0; j4 < 16; ++j4) {
      const int4 e = reinterpret_cast<const int4 *>(patch)[j4];
      const int ee[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) R[4 * j4 + i] = __double_as_longlong(ldexp_i64(R[4 * j4 + i], km + ee[i]));
    }
    __syncwarp();
    store_rows(patch, reinterpret_cast<unsigned long long *>(p.out), p.out_ld, row0, w.m_end, n0c, p.n_valid, hw, R,
               lane);
  } else if constexpr (kMode == kModeKPart) {
    if (m >= p.m_valid) return;
#pragma unroll
    for (int j = 0; j < 64; ++j) {
      const int n = n0c + j;
      if (n < p.n_valid) p.raw[(long long)w.part * p.out_blk + (long long)n * p.out_ld + m] = R[j];
    }
  }
}

// K tiles of a unit are taken in chunks of near-equal length: at most 16 (1024
// products, the exact FP32 range), or 5 in the first exchange GEMM, so that
// three steps of a pass share their accumulators (fewer are drained) and a
// chunk's digit tiles, every CTA streaming its own rows of B, stay in L2 until
// its last pass has read them (5 slices: 122 MB over the chip at 10 K tiles,
// 61 MB at 5).
template <int kMode>
__device__ __forceinline__ int num_chunks(int ktiles) {
  constexpr int most = kMode == kModeX ? kChunkX : kChunkStages;
  return (ktiles + most - 1) / most;
}
__device__ __forceinline__ int chunk_begin(int ktiles, int nch, int c) { return ktiles * c / nch; }

// acc + v 2^sh for 0 <= sh <= 30: one widening multiply-add (2^sh fits a
// signed 32-bit multiplier), exact in int64
__device__ __forceinline__ long long mad_pow2(int v, int pow2, long long acc) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(v), "r"(pow2), "l"(acc));
  return d;
}

// acc + v 2^sh for 32 <= sh <= 63, modulo 2^64: only the high word changes
__device__ __forceinline__ long long add_high(int v, int sh_hi, long long acc) {
  return (long long)((unsigned long long)acc + ((unsigned long long)((uint32_t)v << sh_hi) << 32));
}

__device__ __forceinline__ long long weigh(int v, int sh) {
  const long long x = (long long)v;
  return sh >= 0 ? (x << sh) : ((x + (1ll << (-sh - 1))) >> (-sh));
}

// The passes, sub-passes and steps of one chunk, walked alike by the producer,
// the MMA issuer and the epilogue: groups glo .. ghi share a TMEM buffer,
// steps t0 .. t1-1 (at most 16 / chunk length of them, so that an accumulator
// takes at most 1024 products) accumulate into it, and the sub-pass's first
// step covers every group it touches (glo + first .. ghi).  The longest pass
// comes first: it gives the epilogue the time to store the unit before (240
// atoms: 15.7 ms for the first GEMM, 16.2 ms in the other order).
struct Pass {
  int ghi, glo, t0, t1, first, rmax, q;
  __device__ __forceinline__ void begin(int s, int q_, int len) {
    q = q_;
    rmax = max(1, kChunkStages / len);
    ghi = s - 1;
    t0 = 0;
    set();
  }
  __device__ __forceinline__ bool valid() const { return ghi >= 0; }
  __device__ __forceinline__ void next() {
    t0 = t1;
    if (t0 > ghi) {
      ghi -= q;
      t0 = 0;
    }
    set();
  }
  __device__ __forceinline__ void set() {
    glo = max(0, ghi - q + 1);
    t1 = min(t0 + rmax, ghi + 1);
    first = max(0, t0 - glo);
  }
  // step t: the stacked digits ulo .. ulo + nd - 1 of B, at column tile col of the buffer
  __device__ __forceinline__ void step(int t, int &ulo, int &nd, int &col) const {
    ulo = max(0, glo - t);
    nd = ghi - t - ulo + 1;
    col = t + ulo - glo;
  }
};

// Parameters and operand maps of global unit u: the launch's own (single
// problem) or, in a grouped launch, those of the problem that owns u.
template <bool kGrouped>
__device__ __forceinline__ const SgParams &unit_params(const SgParams &p, const SgGroup &g, int u, int &local,
                                                      int &mol) {
  if (!kGrouped) {
    local = u;
    mol = 0;
    return p;
  }
  int lo = 0, hi = g.nmol - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (g.unit_off[mid] <= u)
      lo = mid;
    else
      hi = mid - 1;
  }
  mol = lo;
  local = u - g.unit_off[lo];
  return g.params[lo];
}

// kHelp: 512 threads, with warps 2, 3 and 12-15 running the Coulomb pass cw (rho
// beside the first exchange GEMM, J beside the second).  The GEMMs leave the
// FP64 pipe and, but for the first one at few orbitals, most of the DRAM rate
// idle; the passes are bound by both, and run on their own or beside the X split
// they were a quarter of a step.
template <int kMode, bool kGrouped, bool kPair, bool kHelp>
__global__ void __launch_bounds__(kHelp ? kThreadsHelp : kThreads, 1)
    slice_gemm_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
                      const __grid_constant__ CUtensorMap tmap_h, const __grid_constant__ CUtensorMap tmap_x, const SgParams p,
                      const SgGroup grp, const CoulombWork cw) {
  constexpr int kRLow = kHelp ? kRegsLowH : kRegsLow, kRHigh = kHelp ? kRegsHighH : kRegsHigh;
  constexpr int NS = ring_stages(kMode, kPair);
  constexpr int SB = stage_bytes(kMode, kPair);
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + NS * SB);
  uint64_t *empty = full + NS;
  uint64_t *acc_full = empty + NS;
  uint64_t *acc_empty = acc_full + kAccBufs;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_empty + kAccBufs);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  uint8_t *patches = smem + NS * SB + kBarBytes;  // modes with row-major stores

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  // CTA pair (the cluster is two neighbours along x): rank 0 issues the MMAs of both CTAs; each CTA loads its own A
  // tile and B tile, drains its own TMEM rows and writes its own output tile.
  const int crank = kPair ? (int)(blockIdx.x & 1u) : 0;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NS; ++i) {
      // pair: rank 0's full barriers count the bytes of both CTAs' copies
      // (rank 0's producer expects them all); rank 1's are not used
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < kAccBufs; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], kPair ? 2 * kEpiWarps : kEpiWarps);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    if (kPair) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                       smem_u32(tmem_slot)),
                   "r"(kTmemCols)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                       smem_u32(tmem_slot)),
                   "r"(kTmemCols)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  // the other CTA's arrivals and commits may target this CTA's barriers from now on
  if (kPair) cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const int total_units = kGrouped ? grp.total : (kPair ? p.npairs : p.nunits);
  const int first_unit = kPair ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
  const int unit_stride = kPair ? (int)(gridDim.x >> 1) : (int)gridDim.x;

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRLow));
    const bool lead = elect_one();
    uint32_t it = 0, st = 0, ph = 1;  // stages filled so far, ring position and the parity of its empty barrier
    bool ok = true, ready = false;
    const uint32_t full0 = kPair ? peer_addr(full, 0) : 0u;
    for (int u = first_unit; u < total_units && ok; u += unit_stride) {
      int lu, mol;
      const SgParams &q = unit_params<kGrouped>(p, grp, u, lu, mol);
      const Unit w = decode_unit<kMode, kPair>(q, lu, crank);
      const CUtensorMap *ma = kGrouped ? &grp.maps[4 * mol] : &tmap_a;
      const CUtensorMap *mb = kGrouped ? &grp.maps[4 * mol + 1] : &tmap_b;
      const CUtensorMap *mh = kGrouped ? &grp.maps[4 * mol + 2] : &tmap_h;
      const int nw = q.nw, hw = nw >> 1, qd = q.q;
      const int nch = num_chunks<kMode>(w.ktiles);
      uint32_t rest = w.kmask;  // sparse: the K tiles of this and the later chunks
      for (int c = 0; c < nch && ok; ++c) {
        const int kb = chunk_begin(w.ktiles, nch, c), ke = chunk_begin(w.ktiles, nch, c + 1);
        Pass ps;
        for (ps.begin(w.s, qd, ke - kb); ps.valid() && ok; ps.next()) {
          for (int t = ps.t0; t < ps.t1 && ok; ++t) {
            int ulo, nd, col;
            ps.step(t, ulo, nd, col);
            // this CTA's part of the nd stacked digits: all of them, or in a pair the
            // first or second half of their rows: `whole` digits from z1 on and, for
            // odd nd, half a digit (before them on rank 1, after them on rank 0)
            const int whole = kPair ? nd >> 1 : nd;
            const bool odd = kPair && (nd & 1);
            const int zh = w.bz0 + (ulo + whole) * w.bzs;
            const int z1 = w.bz0 + (kPair && crank ? ulo + whole + (nd & 1) : ulo) * w.bzs;
            // the first box, and how many whole digits and whether a half follow it
            const bool half_first = odd && (crank || whole == 0);
            const CUtensorMap *m1 = half_first ? mh : mb;
            const int r1 = w.n0 + (half_first && crank ? hw : 0);
            const int zf = half_first ? zh : z1;
            const int more = half_first ? whole : whole - 1;
            const int zm = half_first ? z1 : z1 + w.bzs;
            const uint32_t sb1 = (uint32_t)(kTileBytes + (half_first ? hw : nw) * (2 * kKTile));
            const bool half_last = odd && !half_first;
            const int za = w.az0 + t * w.azs;
            const uint32_t bytes = (uint32_t)(kPair ? 2 * kTileBytes + nd * nw * (2 * kKTile)
                                                    : kTileBytes + nd * nw * (2 * kKTile));
            uint32_t mask = rest;
            for (int kt = kb; kt < ke; ++kt) {
              if (!ready) {
                ok = __all_sync(0xffffffffu, wait_bounded<kPair>(&empty[st], ph, abort_flag, p.status));
                if (!ok) break;
              }
              uint8_t *sa = smem + st * SB;
              uint64_t *fb = &full[st];
              const uint32_t fbr = full0 + st * (uint32_t)sizeof(uint64_t);
              int kc = (w.kt0 + kt) * kKTile;
              if (w.sparse) {
                kc = (__ffs((int)mask) - 1) * kKTile;
                mask &= mask - 1u;
              }
              ++it;
              if (++st == NS) {
                st = 0;
                ph ^= 1u;
              }
              const bool next = mbar_test<kPair>(&empty[st], ph);
              if (lead) {
                // a pair's copies complete on rank 0's barrier
                if (!kPair || crank == 0) mbar_expect_tx(fb, bytes);
                auto copy = [&](uint8_t *dst, const CUtensorMap *map, int row, int z) {
                  if (kPair)
                    tma_load_3d_pair(dst, map, fbr, kc, row, z);
                  else
                    tma_load_3d(dst, map, fb, kc, row, z);
                };
                copy(sa, ma, w.m0, za);
                copy(sa + kTileBytes, m1, r1, zf);
                if (more | (int)half_last) {
                  uint8_t *sb = sa + sb1;
                  for (int d = 0; d < more; ++d) {
                    copy(sb, mb, w.n0, zm + d * w.bzs);
                    sb += nw * (2 * kKTile);
                  }
                  if (half_last) copy(sb, mh, w.n0, zh);
                }
              }
              __syncwarp();
              ready = __all_sync(0xffffffffu, next);
            }
          }
        }
        if (w.sparse)
          for (int kt = kb; kt < ke; ++kt) rest &= rest - 1u;
      }
    }
    if (!ok && crank == 0) {
      // let the copies already issued land before the CTA goes away
      const uint32_t first = it > (uint32_t)NS ? it - NS : 0u;
      for (uint32_t j = first; j < it; ++j)
        wait_bounded<kPair>(&full[j % NS], (j / NS) & 1, abort_flag, p.status, false);
    } else if (!ok) {
      // pair, rank 1: its copies complete on rank 0's barrier, which this
      // CTA cannot wait on; a copy lands within microseconds, so give the
      // ones in flight a fixed 200 us
      const uint64_t t0 = globaltimer_ns();
      while (globaltimer_ns() - t0 < 200000ull) {
      }
    } else if (kPair) {
      // the MMA commits of the last stages arrive from rank 0: let them
      // land before this CTA can leave
      const uint32_t first = it > (uint32_t)NS ? it - NS : 0u;
      for (uint32_t j = first; j < it; ++j)
        wait_bounded<kPair>(&empty[j % NS], (j / NS) & 1, abort_flag, p.status, false);
    }
    __syncwarp();
  } else if (warp == 1) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRLow));
    // pair, rank 1: rank 0's warp issues the MMAs of both CTAs
    if (!kPair || crank == 0) {
    // ------------------------------------------------------------ MMA issuer
    const bool lead = elect_one();
    uint32_t st = 0, ph = 0, buf = 0, bph = 1;  // ring position, accumulator buffer, parities of their barriers
    bool ok = true, ready = false;
    const uint64_t desc0 = sw128_desc(smem_u32(smem));
    for (int u = first_unit; u < total_units && ok; u += unit_stride) {
      int lu, mol;
      const SgParams &q = unit_params<kGrouped>(p, grp, u, lu, mol);
      const Unit w = decode_unit<kMode, kPair>(q, lu, crank);
      const int nw = q.nw, qd = q.q;
      const int nch = num_chunks<kMode>(w.ktiles);
      for (int c = 0; c < nch && ok; ++c) {
        const int kb = chunk_begin(w.ktiles, nch, c), ke = chunk_begin(w.ktiles, nch, c + 1);
        Pass ps;
        for (ps.begin(w.s, qd, ke - kb); ps.valid() && ok; ps.next()) {
          ok = __all_sync(0xffffffffu, wait_bounded<kPair>(&acc_empty[buf], bph, abort_flag, p.status));
          if (!ok) break;
          tc_fence_after();
          for (int t = ps.t0; t < ps.t1 && ok; ++t) {
            int ulo, nd, col;
            ps.step(t, ulo, nd, col);
            const uint32_t idesc = idesc_n(kPair ? kIdesc2 : kIdesc1, nd * nw);
            const uint32_t dt = tmem_base + buf * kAccCols + (uint32_t)(col * nw);
            uint32_t acc = t > ps.t0 ? 1u : 0u;  // the sub-pass's first MMA overwrites its columns
            for (int kt = kb; kt < ke; ++kt) {
              if (!ready) {
                ok = __all_sync(0xffffffffu, wait_bounded<kPair>(&full[st], ph, abort_flag, p.status));
                if (!ok) break;
              }
              tc_fence_after();
              const uint64_t da = desc0 + (uint64_t)(st * (uint32_t)(SB >> 4));
              const uint64_t db = da + (uint64_t)(kTileBytes >> 4);
              uint64_t *eb = &empty[st];
              if (++st == NS) {
                st = 0;
                ph ^= 1u;
              }
              const bool next = mbar_test<kPair>(&full[st], ph);
              if (lead) {
                if (kt + 1 < w.ktiles || w.ksteps_last == kKTile / 16) {
#pragma unroll
                  for (int k = 0; k < kKTile / 16; ++k) {
                    if (kPair)
                      umma_bf16_pair(dt, da + 2 * k, db + 2 * k, idesc, k > 0 ? 1u : acc);
                    else
                      umma_bf16(dt, da + 2 * k, db + 2 * k, idesc, k > 0 ? 1u : acc);
                  }
                } else {
                  for (int k = 0; k < w.ksteps_last; ++k) {
                    if (kPair)
                      umma_bf16_pair(dt, da + 2 * k, db + 2 * k, idesc, k > 0 ? 1u : acc);
                    else
                      umma_bf16(dt, da + 2 * k, db + 2 * k, idesc, k > 0 ? 1u : acc);
                  }
                }
                if (kPair)
                  umma_commit_pair(eb);
                else
                  umma_commit(eb);
              }
              __syncwarp();
              acc = 1u;
              ready = __all_sync(0xffffffffu, next);
            }
          }
          if (!ok) break;
          if (lead) {
            if (kPair)
              umma_commit_pair(&acc_full[buf]);
            else
              umma_commit(&acc_full[buf]);
          }
          __syncwarp();
          buf ^= 1u;
          bph ^= (uint32_t)(buf == 0);
        }
      }
    }
    if (!ok) {
      // wait for the MMAs already issued before the TMEM is released
      uint64_t *done = &acc_full[buf];
      if (lead) {
        if (kPair)
          umma_commit_pair(done);
        else
          umma_commit(done);
      }
      wait_bounded<kPair>(done, bph ^ 1u, abort_flag, p.status, false);
    }
    __syncwarp();
    }
  } else if (warp < kEpiWarp0 || warp >= kEpiWarp0 + kEpiWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRLow));
    if constexpr (kHelp) coulomb_work<kMode == kModeX ? 1 : 2>(cw);
  } else {
    // ------------------------------------------------------------ epilogue
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRHigh));
    const int quad = warp & 3;
    const int half = (warp - kEpiWarp0) >> 2;
    const uint32_t lane_base = tmem_base + ((uint32_t)(quad * 32) << 16);
    // the buffer is handed back to the MMA issuer: this CTA's, or rank 0's in a pair
    const uint32_t acc_empty0 = kPair ? peer_addr(acc_empty, 0) : 0u;
    uint8_t *patch = patches + (warp - kEpiWarp0) * kPatchBytes;
    long long R[64];
    uint32_t buf = 0, bph = 0;
    bool ok = true;
    for (int u = first_unit; u < total_units && ok; u += unit_stride) {
      int lu, mol;
      const SgParams &q = unit_params<kGrouped>(p, grp, u, lu, mol);
      const Unit w = decode_unit<kMode, kPair>(q, lu, crank);
      const int s = w.s, nw = q.nw, hw = nw >> 1, qd = q.q;
      const int T = kMode == kModeRaw ? 0 : q.shiftT[s];
      const int row0 = w.m0 + quad * 32;
      const int m = row0 + lane;
      const int n_base = w.n0 + half * hw;
      const int kexp_base = -14 - 8 * (s - 1) + T;
#pragma unroll
      for (int j = 0; j < 64; ++j) R[j] = 0;
      const int nch = num_chunks<kMode>(w.ktiles);
      for (int c = 0; c < nch && ok; ++c) {
        const int len = chunk_begin(w.ktiles, nch, c + 1) - chunk_begin(w.ktiles, nch, c);
        Pass ps;
        for (ps.begin(s, qd, len); ps.valid() && ok; ps.next()) {
          // one verdict for the warp: its lanes run the aligned loads below together
          ok = __all_sync(0xffffffffu, wait_bounded<kPair>(&acc_full[buf], bph, abort_flag, p.status));
          if (!ok) break;
          tc_fence_after();
          const uint32_t acc0 = lane_base + buf * kAccCols + (uint32_t)(half * hw);
          // 32 (or 16) columns are loaded at a time; a TMEM load takes well under
          // 100 cycles also while MMAs run, a warp's 32 conversions and adds ~550
          // (two warps per scheduler at 16 conversions per clock and SM, the
          // epilogue's floor), so the warps cover each other's loads.
          auto load = [&](int g, int h, uint32_t (&a)[32]) {
            const uint32_t at = acc0 + (uint32_t)((g - ps.glo) * nw + 32 * h);
            if (hw >= 32 * h + 32)
              tmem_ld32(at, a);
            else
              tmem_ld16(at, a);
          };
          auto release = [&]() {
            // the buffer is in registers: hand it back to the MMA warp
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
              if (kPair)
                mbar_arrive_remote(acc_empty0 + buf * (uint32_t)sizeof(uint64_t));
              else
                mbar_arrive(&acc_empty[buf]);
            }
          };
          auto add = [&](int g, auto h_c, const uint32_t (&a)[32]) {
            constexpr int h = decltype(h_c)::value;
            [[maybe_unused]] const int sh = kMode == kModeRaw ? 0 : 8 * (s - 1 - g) - T;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              if (32 * h + 16 * i >= hw) break;
              if constexpr (kMode == kModeRaw) {
                if (m < q.m_valid) {
#pragma unroll
                  for (int j = 0; j < 16; ++j) {
                    const int n = n_base + 32 * h + 16 * i + j;
                    if (n >= q.n_valid) continue;
                    q.raw[((long long)g * q.n_valid + n) * q.m_valid + m] +=
                        (long long)__float2int_rz(__uint_as_float(a[16 * i + j]));
                  }
                }
              } else if (sh >= 0 && sh <= 30) {
                // a weight that fits a 32-bit multiplier: one widening multiply-add
                const int p0 = 1 << sh;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                  long long &r = R[32 * h + 16 * i + j];
                  r = mad_pow2(__float2int_rz(__uint_as_float(a[16 * i + j])), p0, r);
                }
              } else if (sh >= 32) {
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                  long long &r = R[32 * h + 16 * i + j];
                  r = add_high(__float2int_rz(__uint_as_float(a[16 * i + j])), sh - 32, r);
                }
              } else {
                // 2^31, or a low-order group below the kept bits (T > 0): rounded shifts
#pragma unroll
                for (int j = 0; j < 16; ++j)
                  R[32 * h + 16 * i + j] += weigh(__float2int_rz(__uint_as_float(a[16 * i + j])), sh);
              }
            }
          };
          using H0 = std::integral_constant<int, 0>;
          using H1 = std::integral_constant<int, 1>;
          for (int g = ps.glo + ps.first; g <= ps.ghi; ++g) {
            uint32_t a[32];
            load(g, 0, a);
            tmem_wait_ld(a);
            if (hw <= 32 && g == ps.ghi) release();
            add(g, H0{}, a);
            if (hw > 32) {
              load(g, 1, a);
              tmem_wait_ld(a);
              if (g == ps.ghi) release();
              add(g, H1{}, a);
            }
          }
          buf ^= 1u;
          bph ^= (uint32_t)(buf == 0);
        }
      }
      if constexpr (kMode == kModeX) {
        // the exact sums; the X split applies the scales and the rounding to FP64
        if (ok) {
          if (q.rowE) {
            if (lane == 0) tma_store_wait_all();  // the previous unit's stores have left the patch
            __syncwarp();
            const int emax = stage_column_exponents(patch, q.eb, n_base, q.n_valid, hw, lane);
            const int wtop = 8 * (s - 1) - T + 15 + (32 - __clz(q.ktiles * kKTile - 1));
            record_row_bound(q, w, m, hw, wtop, R, kexp_base, patch, emax);
            __syncwarp();
          }
          store_x(patch, kGrouped ? &grp.maps[4 * mol + 3] : &tmap_x, row0, w.m_end, n_base, q.n_valid, hw, R, lane);
        }
      } else if constexpr (kMode != kModeRaw) {
        if (ok) store_tile<kMode>(q, w, m, row0, n_base, hw, R, kexp_base, patch, lane);
      }
    }
    if (kMode == kModeX && lane == 0) tma_store_wait_all();
    __syncwarp();
    // out of tiles: help with what is left of the Coulomb pass
    if constexpr (kHelp) coulomb_work<kMode == kModeX ? 1 : 2>(cw);
  }

  tc_fence_before();
  __syncthreads();
  // neither CTA of a pair frees its TMEM or leaves while the other may still
  // use its barriers, shared memory or accumulators
  if (kPair) cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    if (kPair)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols)
                   : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols)
                   : "memory");
  }
}

// Failure-path self-test of the bounded wait: one thread waits, through the
// pipeline's own wait routine, on an mbarrier that expects an arrival nobody
// makes.  The wait gives up after limit_ns, raises the CTA's abort flag and
// the status bit, and the kernel returns normally (no trap, no fault).
__global__ void wait_selftest_kernel(int *status, unsigned long long limit_ns) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_flag = 0;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (!wait_bounded<false>(&bar, 0, &abort_flag, status, true, limit_ns) && !abort_flag) atomicOr(status, 2);
  }
}

typedef CUresult (*PFN_encodeTiled)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                    const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                    CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                    CUtensorMapFloatOOBfill);

PFN_encodeTiled get_encode_fn() {
  static PFN_encodeTiled fn = nullptr;
  if (!fn) {
    void *ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_encodeTiled>(ptr);
  }
  return fn;
}

}  // namespace

bool make_tmap_bf16(CUtensorMap *map, const void *base, long long k, long long rows, long long planes,
                    long long row_stride_elems, long long plane_stride_elems, int box_rows) {
  PFN_encodeTiled enc = get_encode_fn();
  if (!enc) return false;
  if ((reinterpret_cast<uintptr_t>(base) & 15) || (row_stride_elems * 2) % 16 || (plane_stride_elems * 2) % 16)
    return false;
  cuuint64_t dims[3] = {(cuuint64_t)k, (cuuint64_t)rows, (cuuint64_t)planes};
  cuuint64_t strides[2] = {(cuuint64_t)(row_stride_elems * 2), (cuuint64_t)(plane_stride_elems * 2)};
  cuuint32_t box[3] = {(cuuint32_t)kKTile, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// Tensor map of X's int64 sums [rows][ld] (ld even), boxes of 8 columns x 32 rows, 64B swizzle.
bool make_tmap_x(CUtensorMap *map, const void *base, long long ld, long long rows) {
  PFN_encodeTiled enc = get_encode_fn();
  if (!enc || (reinterpret_cast<uintptr_t>(base) & 15) || (ld & 1)) return false;
  cuuint64_t dims[2] = {(cuuint64_t)ld, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)(ld * 8)};
  cuuint32_t box[2] = {(cuuint32_t)kStoreCols, 32};
  cuuint32_t estr[2] = {1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_INT64, 2, const_cast<void *>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_operand_maps(SgMaps *m, const SgOperand &a, const SgOperand &b, int nw) {
  std::memset(&m->x, 0, sizeof(m->x));
  return make_tmap_bf16(&m->a, a.base, a.k, a.rows, a.planes, a.ld, a.plane_stride, kTile) &&
         make_tmap_bf16(&m->b, b.base, b.k, b.rows, b.planes, b.ld, b.plane_stride, nw) &&
         make_tmap_bf16(&m->h, b.base, b.k, b.rows, b.planes, b.ld, b.plane_stride, nw / 2);
}

void grid_params(SgParams *p, int mode, int M, int N, int K, int s) {
  std::memset(p, 0, sizeof(*p));
  p->mode = mode;
  p->nt_m = (M + kTile - 1) / kTile;
  p->nt_n = (N + kTile - 1) / kTile;
  p->nw = kTile;
  p->q = 2;
  p->nunits = p->nt_m * p->nt_n;
  p->m_valid = M;
  p->n_valid = N;
  p->kvalid = K;
  p->ktiles = (K + kKTile - 1) / kKTile;
  p->s_fixed = s;
  for (int q = 0; q <= 8; ++q) p->shiftT[q] = fixed_point_shift(q, (long long)p->ktiles * kKTile);
}

cudaError_t launch_wait_selftest(int *status, unsigned long long limit_ns, cudaStream_t st) {
  wait_selftest_kernel<<<1, 32, 0, st>>>(status, limit_ns);
  return cudaGetLastError();
}

int slice_gemm_grid(int nunits) {
  static int nsm = 0;
  if (!nsm) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (nsm <= 0) nsm = 1;
  }
  return nunits < nsm ? nunits : nsm;
}

template <int kMode, bool kGrouped, bool kHelp = false>
cudaError_t launch_mode(const SgParams &p, const SgMaps &m, const SgGroup &g, int grid, cudaStream_t st,
                        const CoulombWork &cw = CoulombWork{}) {
  constexpr int smem = smem_bytes(kMode, false);
  auto kern = slice_gemm_kernel<kMode, kGrouped, false, kHelp>;
  static bool attr = false;
  if (!attr) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  kern<<<grid, kHelp ? kThreadsHelp : kThreads, smem, st>>>(m.a, m.b, m.h, m.x, p, g, cw);
  return cudaGetLastError();
}

// CTA-pair launch: clusters of two CTAs, as many clusters as fit at once (at
// most one per tile pair, unless a Coulomb pass wants every SM), persistent over
// the tile pairs; grouped: the tile pairs of several problems (g.total pairs,
// prefix table in pairs).
template <int kMode, bool kGrouped = false, bool kHelp = false>
cudaError_t launch_pair(const SgParams &p, const SgMaps &m, cudaStream_t st, const SgGroup *grp = nullptr,
                        const CoulombWork &cw = CoulombWork{}) {
  auto kern = slice_gemm_kernel<kMode, kGrouped, true, kHelp>;
  constexpr int smem = smem_bytes(kMode, true);
  static int max_clusters = 0;
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.blockDim = dim3(kHelp ? kThreadsHelp : kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (!max_clusters) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    cfg.gridDim = dim3(2 * (unsigned)(slice_gemm_grid(1 << 30) / 2), 1, 1);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n <= 0) {
      cudaGetLastError();
      n = slice_gemm_grid(1 << 30) / 2;
    }
    max_clusters = n > 0 ? n : 1;
  }
  const int np = kGrouped ? grp->total : p.npairs;
  const int nc = np < max_clusters && !kHelp ? np : max_clusters;
  cfg.gridDim = dim3(2 * (unsigned)nc, 1, 1);
  SgGroup g;
  std::memset(&g, 0, sizeof(g));
  if (kGrouped) g = *grp;
  cudaError_t e = cudaLaunchKernelEx(&cfg, kern, m.a, m.b, m.h, m.x, p, g, cw);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

// Row tiles of the first exchange GEMM, `rows` rows each, none across two auxiliary blocks.
static long long x_row_tiles(const SgParams &p, int rows) {
  const long long full = ((long long)kBlock * p.nao + rows - 1) / rows;
  const long long last = (long long)(p.naux - (p.nblk - 1) * kBlock) * p.nao;
  return full * (p.nblk - 1) + (last + rows - 1) / rows;
}

long long slice_gemm_units(const SgParams &p) {
  if (p.mode == kModeX) return x_row_tiles(p, kTile) * p.nt_n;
  if (p.mode == kModeKPart) return (long long)p.nt_m * (p.nt_m + 1) / 2 * p.nblk * p.nsplit;
  if (p.mode == kModeMod)
    return (p.sym ? (long long)p.nt_m * (p.nt_m + 1) / 2 : (long long)p.nt_m * p.nt_n) * p.nblk * p.nsplit;
  return (long long)p.nt_m * p.nt_n;
}

long long slice_gemm_pairs(const SgParams &p) {
  if (p.mode == kModeX) return x_row_tiles(p, 2 * kTile) * p.nt_n;
  if (p.mode == kModeGemm) return (long long)((p.nt_m + 1) / 2) * p.nt_n;
  const long long nt = p.nt_m, na = (nt + 1) / 2;
  if (p.mode == kModeMod && !p.sym) return na * p.nt_n * p.nblk * p.nsplit;
  if (p.mode != kModeKPart && p.mode != kModeMod) return 0;
  return na * (nt - na + 1) * p.nblk * p.nsplit;
}

// Whether a launch runs in CTA-pair mode.  A pair takes in 264 KB per CTA, K
// tile and 5 slices where two single CTAs take 384 KB each, and these kernels
// are bound by the ~70 bytes per clock an SM takes in from L2.  p.pair: 0 never;
// 1 the first exchange GEMM (every tile pair is useful there), and the second
// from 7 tile rows on: its pairs recompute one lower tile per pair of tile rows
// (10 tile rows: 60 tiles for 55, 9.2 ms against 10.1; 5 tile rows: 18 for 15,
// 1.13 ms against 0.99); 2 both wherever they pair.  A stand-alone product pairs
// when every pair has two tiles or there are tiles enough that one more row of
// them does not matter.
static bool use_pairs(const SgParams &p) {
  if (p.mode == kModeMod) return p.pair != 0;
  if (p.mode == kModeGemm) return p.nt_m % 2 == 0 || p.nt_m >= 16;
  if (p.pair == 0) return false;
  return p.mode == kModeX || (p.mode == kModeKPart && (p.pair == 2 || p.nt_m >= 7));
}

void plan_mod_gemm(SgParams *p, int planes, bool sym, bool split) {
  p->nblk = planes;
  p->sym = sym ? 1 : 0;
  const int sms = slice_gemm_grid(1 << 30);
  double best = 0.0;
  int best_pair = 0, best_n = 1;
  for (int pair = 0; pair < 2; ++pair)
    for (int n = 1; n <= (split ? kModSplitMax : 1); ++n) {
      p->nsplit = n;
      const long long workers = pair ? sms / 2 : sms;
      const long long units = pair ? slice_gemm_pairs(*p) : slice_gemm_units(*p);
      if (workers < 1 || (n > 1 && (p->ktiles / n < 16 || units > 8 * workers))) break;
      const double waves = (double)((units + workers - 1) / workers);
      const double cost = waves * ((double)((p->ktiles + n - 1) / n) * (pair ? 370.0 : 515.0) + 3000.0);
      if (best == 0.0 || cost < 0.95 * best) {
        best = cost;
        best_pair = pair;
        best_n = n;
      }
    }
  p->nsplit = best_n;
  p->pair = best_pair;
  p->nunits = (int)slice_gemm_units(*p);
}

cudaError_t launch_slice_gemm(const SgParams &p, const SgMaps &m, cudaStream_t st, const CoulombWork *cw) {
  if (p.nunits <= 0) return cudaSuccess;
  const bool help = cw && cw->kind && (p.mode == kModeX || p.mode == kModeKPart);
  if (use_pairs(p)) {
    const long long np = slice_gemm_pairs(p);
    if (np <= 0 || np > (1ll << 30)) return cudaErrorInvalidValue;
    SgParams q = p;
    q.npairs = (int)np;
    if (p.mode == kModeGemm) return launch_pair<kModeGemm>(q, m, st);
    if (p.mode == kModeMod) return launch_pair<kModeMod>(q, m, st);
    if (help)
      return p.mode == kModeX ? launch_pair<kModeX, false, true>(q, m, st, nullptr, *cw)
                              : launch_pair<kModeKPart, false, true>(q, m, st, nullptr, *cw);
    if (p.mode == kModeX) return launch_pair<kModeX>(q, m, st);
    return launch_pair<kModeKPart>(q, m, st);
  }
  SgGroup g;
  std::memset(&g, 0, sizeof(g));
  if (help) {
    const int all = slice_gemm_grid(1 << 30);
    return p.mode == kModeX ? launch_mode<kModeX, false, true>(p, m, g, all, st, *cw)
                            : launch_mode<kModeKPart, false, true>(p, m, g, all, st, *cw);
  }
  const int grid = slice_gemm_grid(p.nunits);
  switch (p.mode) {
    case kModeX: return launch_mode<kModeX, false>(p, m, g, grid, st);
    case kModeKPart: return launch_mode<kModeKPart, false>(p, m, g, grid, st);
    case kModeRaw: return launch_mode<kModeRaw, false>(p, m, g, grid, st);
    case kModeGemm: return launch_mode<kModeGemm, false>(p, m, g, grid, st);
    case kModeMod: return launch_mode<kModeMod, false>(p, m, g, grid, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_slice_gemm_grouped(int mode, const SgGroup &g, int *status, int grid, cudaStream_t st,
                                      bool pairs) {
  if (g.total <= 0) return cudaSuccess;
  SgParams p;
  std::memset(&p, 0, sizeof(p));
  p.status = status;
  SgMaps dummy;
  std::memset(&dummy, 0, sizeof(dummy));
  if (pairs) {
    if (mode == kModeX) return launch_pair<kModeX, true>(p, dummy, st, &g);
    return cudaErrorInvalidValue;
  }
  const int full_grid = slice_gemm_grid(g.total);
  const int gsz = grid > 0 && grid < full_grid ? grid : full_grid;
  switch (mode) {
    case kModeX: return launch_mode<kModeX, true>(p, dummy, g, gsz, st);
    case kModeKPart: return launch_mode<kModeKPart, true>(p, dummy, g, gsz, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace df
