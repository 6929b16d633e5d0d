// Tensor-core products of the probe for sm_100a: tcgen05.mma with accumulators in tensor
// memory, operands staged in shared memory by TMA, warp-specialised persistent CTA pairs.
//
// Two CTAs on the two SMs of a TPC form a cluster and work on one output tile with cta_group::2
// MMAs: each CTA stages its own 128 rows of the left operand and HALF of the right operand's
// tile, so every byte of the right operand enters and leaves shared memory once per pair instead
// of once per SM.  Four kernels, in this order in the file:
//   tc_kernel            256 x 128 tiles, 320 threads (TMA warp, MMA warp, 8 epilogue warps): the
//                        stand-alone 8-bit and reference products on narrow outputs, and the
//                        two-formats-in-one-pass probe (four accumulators fill tensor memory);
//   tc_gemm_wide_kernel  256 x 256 tiles, two accumulator buffers: stand-alone products on outputs at
//                        least 256 wide;
//   tc_group_kernel      the fused probe (Eq. 3 records of many probes per persistent launch) where several
//                        probes have the same operands: reference L.R and denominator |L|.|R| once per
//                        pair of operands, then the 8-bit products of all its probes, |L| fed to the
//                        MMAs from tensor memory by converter warps, the Eq. 3 statistics reduced in the
//                        epilogue; no M x N matrix ever goes to HBM.  Its comment describes roles and barriers;
//   tc_side_kernel       the same for probes that have their operands to themselves: the three products side by side.
// Common to all: the MMA warp runs its loop converged and one elected lane issues; the epilogue
// warps read the accumulators with tcgen05.ld (a warp may touch the lane quarter warp_id % 4; the
// two warps of a quarter split the columns); a CTA keeps Eq. 3 statistics in registers across tiles
// and writes one record, and the last CTA to finish adds the records up in a fixed order.
//
// Every mbarrier wait is bounded: when one gives up it raises QM_DEVERR_TIMEOUT in the caller's
// error word and flags the CTA, after which every role falls through to the common exit, tensor
// memory is freed and the kernel returns.  No load uses cluster multicast.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <type_traits>
#include <vector>

#include "qm_internal.h"

namespace qm {
namespace {

constexpr int kBlockM = 128;             // rows per CTA
constexpr int kPairM = 256;              // rows per CTA pair
constexpr int kBlockN = 128;             // columns per tile
constexpr int kHalfN = 64;               // right-operand rows staged by each CTA
constexpr int kBlockK = 64;
constexpr int kEpiWarps = 8;
constexpr int kThreads = 64 + 32 * kEpiWarps;                     // 320
constexpr uint32_t kABf16 = kBlockM * kBlockK * 2;                // 16 KB, 128-byte rows
constexpr uint32_t kALp = kBlockM * kBlockK;                      //  8 KB,  64-byte rows
constexpr uint32_t kBBf16 = kHalfN * kBlockK * 2;                 //  8 KB
constexpr uint32_t kBLp = kHalfN * kBlockK;                       //  4 KB
constexpr int kMaxStages = 8;

enum Mode { kLpOnly = 1, kRefOnly = 2, kProbe2 = 3 };

// Stage layout: left-operand tiles first (L, |L|, codes), then the right-operand halves.
template <int MODE> struct Cfg;
// Two 8-bit formats in one pass: the reference and denominator products are shared, each format
// has its own code tiles and its own accumulator.
template <> struct Cfg<kProbe2> {
  static constexpr int kStages = 3;
  static constexpr uint32_t kOffL = 0, kOffLa = kABf16, kOffCl = 2 * kABf16, kOffCl2 = kOffCl + kALp;
  static constexpr uint32_t kOffR = kOffCl2 + kALp, kOffRa = kOffR + kBBf16, kOffCr = kOffRa + kBBf16;
  static constexpr uint32_t kOffCr2 = kOffCr + kBLp;
  static constexpr uint32_t kStageBytes = kOffCr2 + kBLp;         // 72 KB
  static constexpr uint32_t kTmemCols = 512;
};
template <> struct Cfg<kLpOnly> {
  static constexpr int kStages = 8;
  static constexpr uint32_t kOffL = 0, kOffLa = 0, kOffCl = 0, kOffR = 0, kOffRa = 0, kOffCr = kALp;
  static constexpr uint32_t kStageBytes = kALp + kBLp;            // 12 KB
  static constexpr uint32_t kTmemCols = 128;
};
template <> struct Cfg<kRefOnly> {
  static constexpr int kStages = 6;
  static constexpr uint32_t kOffL = 0, kOffLa = 0, kOffCl = 0, kOffR = kABf16, kOffRa = 0, kOffCr = 0;
  static constexpr uint32_t kStageBytes = kABf16 + kBBf16;        // 24 KB
  static constexpr uint32_t kTmemCols = 128;
};

struct KernelArgs {
  int64_t M, N, K;
  int32_t tiles_m, tiles_n, num_tiles;   // tiles of 256 x 128
  const float* dl; int pc_l;             // per-channel flags: delta indexed by batch*M + row
  const float* dr; int pc_r;
  float* out_descaled;                   // LpOnly / RefOnly
  void* out_raw;                         // LpOnly
  double* partials;                      // Probe: gridDim.x records
  uint32_t* done_counter;                // Probe: zero on entry
  qm_metric_result* result;              // Probe
  uint64_t count;                        // Probe: batch * M * N
  uint32_t* err_word;
  uint32_t idesc_lp;                     // instruction descriptor of the 8-bit MMA
  // Probe2: scales and descriptor of the second format (granularities are shared); its record
  // is result[1] and its per-CTA records follow the first format's gridDim.x records
  const float* dl2; const float* dr2;
  uint32_t idesc_lp2;
};

// ------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// shared::cluster address of `addr` (a shared::cta address of this CTA) in CTA `rank`
__device__ __forceinline__ uint32_t map_to_cta(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync() { cluster_arrive(); cluster_wait(); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
// arrive on a barrier given by its shared::cluster address (own CTA or the peer)
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  // default semantics (release at CTA scope): the data this barrier orders lives in tensor
  // memory and is fenced by tcgen05.fence; a cluster-scope release costs a long memory fence
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok;
}
__device__ __forceinline__ uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait.  Returns false when the CTA has been flagged or the time limit (1 s) ran out;
// in the second case it flags the CTA and the caller's error word.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag,
                                          uint32_t* err_word) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_timer_ns();
  uint32_t polls = 0;
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((++polls & 0xffu) == 0) {
      if (*abort_flag) return false;
      if (global_timer_ns() - t0 > 1000000000ull) {
        *abort_flag = 1u;
        if (err_word) atomicOr(err_word, QM_DEVERR_TIMEOUT);
        return false;
      }
    }
  }
}

// The same for a converged warp: every lane waits, and all lanes take the same decision.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag,
                                               uint32_t* err_word) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, err_word));
}

// Tile load into this CTA's shared memory; the byte count is credited to the barrier at
// `bar_cluster_addr`, which may live in the peer CTA (cta_group::2 form).
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar_cluster_addr,
                                            int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar_cluster_addr), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// One lane of a fully converged warp.  The MMA warp runs its whole loop (waits, descriptor
// arithmetic, loop control) convergently and narrows to one lane only around each tcgen05
// instruction: issued from a loop that a single lane runs alone, every MMA cost about 100 cycles
// of issue time, which was the limit of the main loop; issued this way it costs about 60.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.u32 %0, 1, 0, P;\n\t}" : "=r"(p));
  return p != 0;
}

// Arrive on the barrier at this shared-memory offset in BOTH CTAs of the pair once all MMAs
// issued so far have completed.  Called by a converged warp; one lane issues.
__device__ __forceinline__ void tc_commit_pair(uint32_t bar, bool lead) {
  if (!lead) return;
  const uint16_t mask = 3;
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
      ::"r"(bar), "h"(mask) : "memory");
}

// Shared-memory matrix descriptor, contraction-major tile whose rows are exactly one swizzle
// span wide (128 bytes for the bf16 tiles, 64 bytes for the code tiles): eight consecutive rows
// form one swizzle atom, atoms follow each other every 8 * span bytes ("stride byte offset").
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t span_bytes) {
  const uint64_t layout = span_bytes == 128 ? 2ull : (span_bytes == 64 ? 4ull : 6ull);
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3ffffu) >> 4);                      // start address / 16
  d |= (uint64_t)1 << 16;                                       // leading byte offset (unused here)
  d |= (uint64_t)((8u * span_bytes) >> 4) << 32;                // stride byte offset / 16
  d |= (uint64_t)1 << 46;                                       // descriptor version of sm_100
  d |= layout << 61;                                            // swizzle mode
  return d;
}

// The same without its address, and for tiles stored the other way round: contraction-major tiles as above; mn-major
// ones, staged from operands whose contraction is strided (a row of `span` bytes, 32, 64 or 128, holds consecutive operand rows at one contraction entry, swizzled over its
// span) have eight contraction entries per atom, atoms following each other every 8 * span bytes along the contraction and
// every `next` bytes along the operand's rows.  `step` is what a 32-byte-deep (16 bf16, 32 codes) MMA step adds to the
// address field.
struct TileDesc {
  uint32_t hi, lo, step;
  __device__ __forceinline__ uint64_t at(uint32_t addr, int k) const {
    uint64_t d;
    const uint32_t l = ((addr & 0x3ffffu) >> 4) + lo + step * (uint32_t)k;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(l), "r"(hi));
    return d;
  }
};
__device__ __forceinline__ TileDesc tile_desc(bool mn_major, uint32_t span, uint32_t entries_per_step, uint32_t next) {
  TileDesc d;
  const uint64_t full = smem_desc(0u, span);
  d.hi = (uint32_t)(full >> 32);
  d.lo = mn_major ? (next >> 4) << 16 : 1u << 16;
  d.step = mn_major ? entries_per_step * span / 16u : 2u;
  return d;
}
// bits of the instruction descriptor for operands whose tiles in shared memory are mn-major
constexpr uint32_t kIdescMnMajorA = 1u << 15, kIdescMnMajorB = 1u << 16;

enum MmaKind { kKindF16 = 0, kKindF8 = 1, kKindI8 = 2 };

// D[256 x N] (+)= A[256 x k] . B[N x k]^T across the CTA pair; called by a converged warp of the
// leader, one lane issues.
template <int KIND>
__device__ __forceinline__ void mma_pair(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc,
                                         uint32_t accumulate, bool lead) {
  if (!lead) return;
  if (KIND == kKindF16) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(accumulate) : "memory");
  } else if (KIND == kKindF8) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(accumulate) : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::i8 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(accumulate) : "memory");
  }
}

// 32 lanes x 32 consecutive 32-bit columns: thread t of the warp gets lane (base lane + t).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
        "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
        "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Instruction descriptor: D format [4,6), A format [7,10), B format [10,13), majors [15],[16]
// (0 = contraction-major), N/8 at [17,23), M/16 at [24,29).
__host__ __device__ constexpr uint32_t make_idesc(uint32_t c_fmt, uint32_t a_fmt, uint32_t b_fmt,
                                                  uint32_t m, uint32_t n) {
  return (c_fmt << 4) | (a_fmt << 7) | (b_fmt << 10) | ((n >> 3) << 17) | ((m >> 4) << 24);
}

struct alignas(16) Shared {
  uint64_t full[kMaxStages];     // used in the leader CTA: both CTAs' loads of a stage have landed
  uint64_t empty[kMaxStages];    // per CTA: the pair's MMAs have finished reading the stage
  uint64_t tmem_full;            // per CTA: the tile's accumulators are complete
  uint64_t tmem_empty;           // leader: both CTAs' epilogues have drained the accumulators
  uint64_t lp_done;              // leader (probe): both CTAs' epilogues have finished a tile
  uint32_t tmem_base;
  uint32_t abort_flag;
  uint32_t is_last;
  uint32_t pad;
  float delta_r[2][kBlockN];
  float delta_r2[2][kBlockN];    // Probe2: column scales of the second format
  double red[10][kEpiWarps];
};

// Named barrier 1 over the 256 epilogue threads, returning the OR of `flag` over all of them.
__device__ __forceinline__ bool epi_barrier_any(bool flag) {
  uint32_t out;
  __syncwarp();            // bar.red wants the whole warp, whose lanes have waited on a barrier one by one
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\t"
      "bar.red.or.pred p, 1, 256, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(out)
      : "r"((uint32_t)flag)
      : "memory");
  return out != 0;
}

struct TileCoord { int m_tile, n_tile, b; };
__device__ __forceinline__ TileCoord tile_coord(int t, const KernelArgs& a) {
  TileCoord c;
  const int per_b = a.tiles_m * a.tiles_n;
  c.b = t / per_b;
  const int r = t - c.b * per_b;
  c.m_tile = r / a.tiles_n;
  c.n_tile = r - c.m_tile * a.tiles_n;
  return c;
}

// 32 lanes x 16 consecutive 32-bit columns.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15])
      : "r"(taddr)
      : "memory");
}

// Two-wide fp32 arithmetic (one instruction for a pair of values).
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t x, uint64_t y, uint64_t z) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(x), "l"(y), "l"(z));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t x, uint64_t y) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t x, uint64_t y) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
  return r;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float max3(float x, float y, float z) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(x), "f"(y), "f"(z));
  return r;
}

// Eq. 3 statistics of one row, kept two-wide across the columns of a tile.
struct Stats2 {
  uint64_t be, d2, r2, n2;
  float mx;
};

// 16 consecutive columns of one row: reference rc, denominator rd, raw 8-bit accumulator rq.
// ndl2 holds (-delta_l, -delta_l); dr_s points at the 16 column scales (per_col) or is unused.
// n_live < 16 only in the last, ragged column chunk of a matrix.
template <int LPKIND, bool RAGGED>
__device__ __forceinline__ void stats16(const uint32_t* rc, const uint32_t* rd, const uint32_t* rq,
                                        uint64_t ndl2, const float* dr_s, bool per_col, uint64_t dr_tensor2,
                                        int n_live, Stats2& s) {
#pragma unroll
  for (int j = 0; j < 16; j += 2) {
    const bool live0 = !RAGGED || j < n_live, live1 = !RAGGED || j + 1 < n_live;
    const float a0 = LPKIND == kKindI8 ? (float)(int)rq[j] : __uint_as_float(rq[j]);
    const float a1 = LPKIND == kKindI8 ? (float)(int)rq[j + 1] : __uint_as_float(rq[j + 1]);
    const uint64_t dr2 = per_col ? *reinterpret_cast<const uint64_t*>(dr_s + j) : dr_tensor2;
    float c0 = __uint_as_float(rc[j]), c1 = __uint_as_float(rc[j + 1]);
    float d0 = __uint_as_float(rd[j]), d1 = __uint_as_float(rd[j + 1]);
    if (!live0) { c0 = 0.f; d0 = 0.f; }
    if (!live1) { c1 = 0.f; d1 = 0.f; }
    const uint64_t cv2 = pack2(c0, c1), dd2 = pack2(d0, d1);
    uint64_t diff2 = fma2(mul2(pack2(live0 ? a0 : 0.f, live1 ? a1 : 0.f), ndl2), dr2, cv2);   // C - A dl dr
    float e0, e1;
    unpack2(diff2, e0, e1);
    // D == 0 implies C == Q == 0, so clamping the divisor keeps BE = 0 there without a branch
    const float r0 = rcp_approx(fmaxf(d0, 1e-37f)), r1 = rcp_approx(fmaxf(d1, 1e-37f));
    const uint64_t be2 = mul2(pack2(fabsf(e0), fabsf(e1)), pack2(r0, r1));
    float b0, b1;
    unpack2(be2, b0, b1);
    s.be = add2(s.be, be2);
    s.mx = max3(s.mx, b0, b1);
    s.d2 = fma2(diff2, diff2, s.d2);
    s.r2 = fma2(cv2, cv2, s.r2);
    s.n2 = fma2(dd2, dd2, s.n2);
  }
}

// 32 rows x 32 columns of output from a warp that holds a row per lane: through 4 KB of shared memory (16-byte
// units permuted with the row: conflict-free both ways), so that every store instruction writes whole
// 128-byte lines.  A row per thread puts the 32 lanes of a store on 32 lines, sixteen bytes each; with
// short contractions those stores, not the MMAs, were what a tile took: 4096 x 3072 x 768 42 us, staged 20.
// Outputs whose rows do not all start on 16 bytes are written a column per lane.
__device__ __forceinline__ void store_chunk(uint4* stage, int lane, const uint32_t (&r)[32], uint32_t* out, int64_t ld, int rows,
                                            int cols, bool vec_ok) {
#pragma unroll
  for (int j = 0; j < 8; ++j) stage[lane * 8 + (j ^ (lane & 7))] = make_uint4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
  __syncwarp();
  if (cols == 32 && vec_ok) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int row = 4 * i + (lane >> 3), u = lane & 7;
      if (row < rows) *reinterpret_cast<uint4*>(out + row * ld + 4 * u) = stage[row * 8 + (u ^ (row & 7))];
    }
  } else {
    const uint32_t* w = reinterpret_cast<const uint32_t*>(stage);
    for (int row = 0; row < rows; ++row)
      if (lane < cols) out[row * ld + lane] = w[row * 32 + (((lane >> 2) ^ (row & 7)) << 2) + (lane & 3)];
  }
  __syncwarp();
}

template <int MODE, int LPKIND, int LPKIND2>
__global__ void __launch_bounds__(kThreads, 1)
tc_kernel(const __grid_constant__ CUtensorMap map_l, const __grid_constant__ CUtensorMap map_r,
          const __grid_constant__ CUtensorMap map_la, const __grid_constant__ CUtensorMap map_ra,
          const __grid_constant__ CUtensorMap map_cl, const __grid_constant__ CUtensorMap map_cr,
          const __grid_constant__ CUtensorMap map_cl2, const __grid_constant__ CUtensorMap map_cr2,
          const KernelArgs a) {
  constexpr bool kAnyProbe = MODE == kProbe2;
  constexpr int kFormats = MODE == kProbe2 ? 2 : 1;
  using C = Cfg<MODE>;
  constexpr int kStages = C::kStages;
  extern __shared__ uint8_t smem_raw[];
  // tiles start on a 1024-byte boundary (the 128-byte swizzle atom); the offset is the same in
  // both CTAs of the pair because their dynamic shared memory starts at the same address
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  Shared* sh = reinterpret_cast<Shared*>(tiles + (size_t)kStages * C::kStageBytes);

  // known to the compiler to be the same in all lanes (see tc_group_kernel)
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();                   // 0 = leader
  const int pair = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;
  const int num_kb = (int)((a.K + kBlockK - 1) / kBlockK);
  volatile uint32_t* abort_flag = &sh->abort_flag;

  if (warp == 0 && lane < 8) {
    // fetch the tensor maps into the descriptor cache while the CTA sets itself up
    const CUtensorMap* maps[8] = {&map_l, &map_r, &map_la, &map_ra, &map_cl, &map_cr, &map_cl2, &map_cr2};
    asm volatile("prefetch.tensormap [%0];" ::"l"(maps[lane]) : "memory");
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&sh->full[s]), 1);
      mbar_init(smem_u32(&sh->empty[s]), 1);
    }
    mbar_init(smem_u32(&sh->tmem_full), 1);
    mbar_init(smem_u32(&sh->tmem_empty), 2 * kEpiWarps);
    mbar_init(smem_u32(&sh->lp_done), 2 * kEpiWarps);
    sh->abort_flag = 0;
    sh->is_last = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&sh->tmem_base)), "r"(C::kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();          // the peer's barriers and tensor memory exist before anyone uses them
  pdl_prologue();          // everything above overlapped the tail of the previous kernel
  tc_fence_after();
  const uint32_t tmem_base = sh->tmem_base;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (both CTAs)
    if (lane == 0) {
      uint32_t g = 0;                                           // running k-block count
      bool ok = true;
      for (int t = pair; t < a.num_tiles && ok; t += num_pairs) {
        const TileCoord tc = tile_coord(t, a);
        const int r0 = tc.m_tile * kPairM + (int)rank * kBlockM;     // this CTA's left-operand rows
        const int c0 = tc.n_tile * kBlockN + (int)rank * kHalfN;     // this CTA's half of the right operand
        for (int kb = 0; kb < num_kb; ++kb, ++g) {
          const int s = g % kStages;
          const uint32_t use = g / kStages;
          if (use > 0 && !mbar_wait(smem_u32(&sh->empty[s]), (use - 1) & 1, abort_flag, a.err_word)) {
            ok = false;
            break;
          }
          // one barrier (the leader's) collects the bytes of both CTAs
          if (rank == 0) mbar_expect_tx(smem_u32(&sh->full[s]), 2 * C::kStageBytes);
          const uint32_t bar = map_to_cta(smem_u32(&sh->full[s]), 0);
          const uint32_t base = smem_u32(tiles + (size_t)s * C::kStageBytes);
          const int k0 = kb * kBlockK;
          if (kAnyProbe || MODE == kRefOnly) {
            tma_load_3d(base + C::kOffL, &map_l, bar, k0, r0, tc.b);
            tma_load_3d(base + C::kOffR, &map_r, bar, k0, c0, tc.b);
          }
          if (kAnyProbe) {
            tma_load_3d(base + C::kOffLa, &map_la, bar, k0, r0, tc.b);
            tma_load_3d(base + C::kOffRa, &map_ra, bar, k0, c0, tc.b);
          }
          if (kAnyProbe || MODE == kLpOnly) {
            tma_load_3d(base + C::kOffCl, &map_cl, bar, k0, r0, tc.b);
            tma_load_3d(base + C::kOffCr, &map_cr, bar, k0, c0, tc.b);
          }
          if constexpr (MODE == kProbe2) {
            tma_load_3d(base + C::kOffCl2, &map_cl2, bar, k0, r0, tc.b);
            tma_load_3d(base + C::kOffCr2, &map_cr2, bar, k0, c0, tc.b);
          }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (leader CTA only)
    if (rank == 0) {   // the whole warp, converged: see elect_one()
      const bool lead = elect_one();
      constexpr uint32_t idesc_bf16 = make_idesc(1, 1, 1, kPairM, kBlockN);
      uint32_t g = 0, it = 0;
      bool ok = true;
      for (int t = pair; t < a.num_tiles && ok; t += num_pairs, ++it) {
        const uint32_t col_ref = 0u, col_den = 128u;
        const uint32_t col_lp = MODE == kProbe2 ? 256u : 0u;
        auto issue_ref = [&](uint32_t base, int kb) {
          const uint64_t dl = smem_desc(base + C::kOffL, 128), dr = smem_desc(base + C::kOffR, 128);
#pragma unroll
          for (int k = 0; k < kBlockK / 16; ++k)   // 16 bf16 = 32 bytes = 2 descriptor units per step
            mma_pair<kKindF16>(tmem_base + col_ref, dl + 2 * k, dr + 2 * k, idesc_bf16, (kb | k) != 0, lead);
        };
        auto issue_den = [&](uint32_t base, int kb) {
          const uint64_t dl = smem_desc(base + C::kOffLa, 128), dr = smem_desc(base + C::kOffRa, 128);
#pragma unroll
          for (int k = 0; k < kBlockK / 16; ++k)
            mma_pair<kKindF16>(tmem_base + col_den, dl + 2 * k, dr + 2 * k, idesc_bf16, (kb | k) != 0, lead);
        };
        auto issue_lp = [&](uint32_t base, int kb) {
          const uint64_t dl = smem_desc(base + C::kOffCl, 64), dr = smem_desc(base + C::kOffCr, 64);
#pragma unroll
          for (int k = 0; k < kBlockK / 32; ++k)   // 32 codes = 32 bytes per step
            mma_pair<LPKIND>(tmem_base + col_lp, dl + 2 * k, dr + 2 * k, a.idesc_lp, (kb | k) != 0, lead);
        };
        // Probe2: the second format's accumulator takes the fourth block (columns 384..511), so
        // nothing rotates.  The reference and denominator blocks come back when both epilogues
        // have copied them out (tmem_empty), the two 8-bit blocks when they have finished the tile
        // (lp_done); the reference and denominator MMAs of as many k-blocks as there are stages
        // are therefore issued between the two signals.
        auto issue_lp2 = [&](uint32_t base, int kb) {
          if constexpr (MODE == kProbe2) {
            const uint64_t dl = smem_desc(base + C::kOffCl2, 64), dr = smem_desc(base + C::kOffCr2, 64);
#pragma unroll
            for (int k = 0; k < kBlockK / 32; ++k)
              mma_pair<LPKIND2>(tmem_base + 384u, dl + 2 * k, dr + 2 * k, a.idesc_lp2, (kb | k) != 0, lead);
          }
        };
        int kb = 0;
        if (MODE == kProbe2) {
          if (it > 0 && !mbar_wait_warp(smem_u32(&sh->tmem_empty), (it - 1) & 1, abort_flag, a.err_word)) break;
          tc_fence_after();
          const int n_ahead = num_kb < kStages ? num_kb : kStages;
          for (int j = 0; j < n_ahead && ok; ++j) {
            const int s = (g + j) % kStages;
            if (!mbar_wait_warp(smem_u32(&sh->full[s]), ((g + j) / kStages) & 1, abort_flag, a.err_word)) ok = false;
            tc_fence_after();
            if (ok) {
              const uint32_t base = smem_u32(tiles + (size_t)s * C::kStageBytes);
              issue_ref(base, j);
              issue_den(base, j);
            }
          }
          if (!ok) break;
          if (it > 0 && !mbar_wait_warp(smem_u32(&sh->lp_done), (it - 1) & 1, abort_flag, a.err_word)) break;
          tc_fence_after();
          for (; kb < n_ahead; ++kb, ++g) {
            const int s = g % kStages;
            const uint32_t base = smem_u32(tiles + (size_t)s * C::kStageBytes);
            issue_lp(base, kb);
            issue_lp2(base, kb);
            tc_commit_pair(smem_u32(&sh->empty[s]), lead);
          }
        }
        if (MODE != kProbe2 && it > 0 &&
            !mbar_wait_warp(smem_u32(&sh->tmem_empty), (it - 1) & 1, abort_flag, a.err_word))
          break;
        tc_fence_after();
        for (; kb < num_kb; ++kb, ++g) {
          const int s = g % kStages;
          const uint32_t use = g / kStages;
          if (!mbar_wait_warp(smem_u32(&sh->full[s]), use & 1, abort_flag, a.err_word)) { ok = false; break; }
          tc_fence_after();
          const uint32_t base = smem_u32(tiles + (size_t)s * C::kStageBytes);
          if (kAnyProbe || MODE == kRefOnly) issue_ref(base, kb);
          if (kAnyProbe) issue_den(base, kb);
          if (kAnyProbe || MODE == kLpOnly) issue_lp(base, kb);
          issue_lp2(base, kb);
          tc_commit_pair(smem_u32(&sh->empty[s]), lead);        // frees the stage in both CTAs
        }
        if (ok) tc_commit_pair(smem_u32(&sh->tmem_full), lead); // this tile's accumulators are complete
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue (warps 2..9, both CTAs)
    const int q = warp & 3;                       // tensor-memory lane quarter this warp may read
    const int h = (warp - 2) >> 2;                // which 64-column half of the tile
    const int et = (warp - 2) * 32 + lane;        // 0..255
    const float dl_tensor = (MODE != kRefOnly && !a.pc_l) ? __ldg(a.dl) : 1.f;
    const float dr_tensor = (MODE != kRefOnly && !a.pc_r) ? __ldg(a.dr) : 1.f;
    const bool per_col = MODE != kRefOnly && a.pc_r;
    const uint32_t tmem_empty_leader = map_to_cta(smem_u32(&sh->tmem_empty), 0);
    double acc[kFormats][5];                       // per format: sum BE, max BE, sum diff^2, sum C^2, sum D^2
#pragma unroll
    for (int f = 0; f < kFormats; ++f)
#pragma unroll
      for (int i = 0; i < 5; ++i) acc[f][i] = 0.0;
    [[maybe_unused]] const float dl_tensor2 = (MODE == kProbe2 && !a.pc_l) ? __ldg(a.dl2) : 1.f;
    [[maybe_unused]] const float dr_tensor2 = (MODE == kProbe2 && !a.pc_r) ? __ldg(a.dr2) : 1.f;
    auto add_stats = [&](int f, const Stats2& st) {
      float x0, x1;
      unpack2(st.be, x0, x1); acc[f][0] += (double)x0 + (double)x1;
      unpack2(st.d2, x0, x1); acc[f][2] += (double)x0 + (double)x1;
      unpack2(st.r2, x0, x1); acc[f][3] += (double)x0 + (double)x1;
      unpack2(st.n2, x0, x1); acc[f][4] += (double)x0 + (double)x1;
      acc[f][1] = fmax(acc[f][1], (double)st.mx);
    };
    uint32_t it = 0;
    for (int t = pair; t < a.num_tiles; t += num_pairs, ++it) {
      const TileCoord tc = tile_coord(t, a);
      float* dr_s = sh->delta_r[it & 1];
      [[maybe_unused]] float* dr_s2 = sh->delta_r2[it & 1];
      if (per_col && et < kBlockN) {
        const int64_t col = (int64_t)tc.n_tile * kBlockN + et;
        dr_s[et] = col < a.N ? __ldg(a.dr + (int64_t)tc.b * a.N + col) : 0.f;
        if (MODE == kProbe2) dr_s2[et] = col < a.N ? __ldg(a.dr2 + (int64_t)tc.b * a.N + col) : 0.f;
      }
      const int64_t row = (int64_t)tc.m_tile * kPairM + rank * kBlockM + q * 32 + lane;
      const bool row_ok = row < a.M;
      float dlv = dl_tensor;
      if (MODE != kRefOnly && a.pc_l) dlv = row_ok ? __ldg(a.dl + (int64_t)tc.b * a.M + row) : 0.f;
      [[maybe_unused]] float dlv2 = dl_tensor2;
      if (MODE == kProbe2 && a.pc_l) dlv2 = row_ok ? __ldg(a.dl2 + (int64_t)tc.b * a.M + row) : 0.f;

      const bool ok = mbar_wait(smem_u32(&sh->tmem_full), it & 1, abort_flag, a.err_word);
      // one barrier publishes delta_r and makes the give-up decision uniform over the epilogue
      if (epi_barrier_any(!ok)) break;
      tc_fence_after();
      const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
      if (MODE == kProbe2) {
        // Fixed blocks: reference 0, denominator 128, first format 256, second format 384.  Copy
        // this warp's 64 reference and denominator columns into registers and hand those two
        // blocks back (the next tile's reference and denominator MMAs start), walk both 8-bit
        // blocks in chunks of 16 columns, then report the tile finished (lp_done).
        const int64_t colw = (int64_t)tc.n_tile * kBlockN + h * 64;
        uint32_t rc[64], rd[64], rq[16];
        tmem_ld32(lane_addr + 0u + h * 64, *reinterpret_cast<uint32_t(*)[32]>(&rc[0]));
        tmem_ld32(lane_addr + 0u + h * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&rc[32]));
        tmem_ld32(lane_addr + 128u + h * 64, *reinterpret_cast<uint32_t(*)[32]>(&rd[0]));
        tmem_ld32(lane_addr + 128u + h * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&rd[32]));
        tmem_ld_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(tmem_empty_leader);
        Stats2 st{0ull, 0ull, 0ull, 0ull, 0.f}, st2{0ull, 0ull, 0ull, 0ull, 0.f};
        const uint64_t ndl2 = pack2(-dlv, -dlv), drt2 = pack2(dr_tensor, dr_tensor);
        const uint64_t ndl2b = pack2(-dlv2, -dlv2), drt2b = pack2(dr_tensor2, dr_tensor2);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int cc0 = h * 64 + c * 16;
          const int64_t col0 = colw + c * 16;
          if (col0 < a.N) {                       // uniform across the warp
            const int n_live = (int)(a.N - col0 < 16 ? a.N - col0 : 16);
            tmem_ld16(lane_addr + 256u + cc0, rq);
            tmem_ld_wait();
            if (n_live == 16) stats16<LPKIND, false>(&rc[c * 16], &rd[c * 16], rq, ndl2, dr_s + cc0, per_col, drt2, 16, st);
            else stats16<LPKIND, true>(&rc[c * 16], &rd[c * 16], rq, ndl2, dr_s + cc0, per_col, drt2, n_live, st);
            tmem_ld16(lane_addr + 384u + cc0, rq);
            tmem_ld_wait();
            if (n_live == 16) stats16<LPKIND2, false>(&rc[c * 16], &rd[c * 16], rq, ndl2b, dr_s2 + cc0, per_col, drt2b, 16, st2);
            else stats16<LPKIND2, true>(&rc[c * 16], &rd[c * 16], rq, ndl2b, dr_s2 + cc0, per_col, drt2b, n_live, st2);
          }
        }
        if (row_ok) {
          add_stats(0, st);
          if constexpr (kFormats == 2) add_stats(1, st2);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(map_to_cta(smem_u32(&sh->lp_done), 0));
      } else {
        uint4* const stage = reinterpret_cast<uint4*>(sh + 1) + (warp - 2) * 256;      // 4 KB per epilogue warp
        const int64_t row0 = row - lane;
        const int rows_live = (int)(a.M - row0 < 32 ? a.M - row0 : 32);      // <= 0: none
        const bool vec_ok = (a.N & 3) == 0 && (reinterpret_cast<uintptr_t>(a.out_descaled) & 15) == 0 &&
                            (reinterpret_cast<uintptr_t>(a.out_raw) & 15) == 0;
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
          const int cc0 = h * 64 + c * 32;          // first column of this chunk inside the tile
          const int64_t col0 = (int64_t)tc.n_tile * kBlockN + cc0;
          if (col0 >= a.N) break;                   // uniform across the warp
          const int n_live = (int)(a.N - col0 < 32 ? a.N - col0 : 32);
          uint32_t r[32];
          tmem_ld32(lane_addr + cc0, r);
          tmem_ld_wait();
          const int64_t o0 = ((int64_t)tc.b * a.M + row0) * a.N + col0;
          if (MODE == kRefOnly) {
            store_chunk(stage, lane, r, reinterpret_cast<uint32_t*>(a.out_descaled) + o0, a.N, rows_live, n_live, vec_ok);
          } else {
            if (a.out_raw) store_chunk(stage, lane, r, reinterpret_cast<uint32_t*>(a.out_raw) + o0, a.N, rows_live, n_live, vec_ok);
            if (a.out_descaled) {
#pragma unroll
              for (int j = 0; j < 32; ++j) {
                const float acc = LPKIND == kKindI8 ? (float)(int)r[j] : __uint_as_float(r[j]);
                r[j] = __float_as_uint(acc * (dlv * (per_col ? dr_s[cc0 + j] : dr_tensor)));
              }
              store_chunk(stage, lane, r, reinterpret_cast<uint32_t*>(a.out_descaled) + o0, a.N, rows_live, n_live, vec_ok);
            }
          }
        }
      }
      if (!kAnyProbe) {
        // this warp has finished reading the accumulator of the tile: tell the leader's MMA lane
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(tmem_empty_leader);
      }
    }
    if (kAnyProbe) {
      // per format: warp sums -> CTA record -> (last CTA) fixed-order sum of all records
#pragma unroll
      for (int f = 0; f < kFormats; ++f) {
#pragma unroll
        for (int i = 0; i < 5; ++i) {
          double x = acc[f][i];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            const double y = __shfl_xor_sync(0xffffffffu, x, o);
            x = i == 1 ? fmax(x, y) : x + y;
          }
          if (lane == 0) sh->red[f * 5 + i][warp - 2] = x;
        }
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (et == 0) {
        for (int f = 0; f < kFormats; ++f) {
          double* rec = a.partials + ((int64_t)f * gridDim.x + blockIdx.x) * kPartialDoubles;
          for (int i = 0; i < 5; ++i) {
            double x = 0.0;
            for (int w = 0; w < kEpiWarps; ++w) x = i == 1 ? fmax(x, sh->red[f * 5 + i][w]) : x + sh->red[f * 5 + i][w];
            __stcg(rec + i, x);
          }
        }
        __threadfence();
        const uint32_t prev = atomicAdd(a.done_counter, 1u);
        sh->is_last = prev == gridDim.x - 1 ? 1u : 0u;
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (sh->is_last && warp == 2) {
        // last CTA: every record is visible; fixed-order sum (lane l takes records l, l+32, ...)
        __threadfence();
        for (int f = 0; f < kFormats; ++f) {
          double r[5] = {0, 0, 0, 0, 0};
          for (int i = lane; i < (int)gridDim.x; i += 32) {
            const double* rec = a.partials + ((int64_t)f * gridDim.x + i) * kPartialDoubles;
            r[0] += __ldcg(rec); r[1] = fmax(r[1], __ldcg(rec + 1)); r[2] += __ldcg(rec + 2);
            r[3] += __ldcg(rec + 3); r[4] += __ldcg(rec + 4);
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            r[0] += __shfl_xor_sync(0xffffffffu, r[0], o);
            r[1] = fmax(r[1], __shfl_xor_sync(0xffffffffu, r[1], o));
            r[2] += __shfl_xor_sync(0xffffffffu, r[2], o);
            r[3] += __shfl_xor_sync(0xffffffffu, r[3], o);
            r[4] += __shfl_xor_sync(0xffffffffu, r[4], o);
          }
          if (lane == 0) {
            qm_metric_result* out = a.result + f;
            out->sum_be = r[0]; out->max_be = r[1]; out->sum_diff2 = r[2];
            out->sum_ref2 = r[3]; out->sum_den2 = r[4];
            out->count = a.count;
            out->device_error = a.err_word ? *reinterpret_cast<volatile uint32_t*>(a.err_word) : 0u;
            out->reserved = 0;
          }
        }
      }
    }
  }

  // ---------------------------------------------------------------- common exit
  // Neither CTA may leave while the other can still read its shared memory, signal its
  // barriers or write its tensor memory.
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(C::kTmemCols)
                 : "memory");
  }
}

// ------------------------------------------------------------------ plain products on 256 x 256 tiles
// qm_gemm and qm_gemm_ref on wide outputs.  One accumulator per tile leaves room for 256-column
// tiles, which halves the MMA instructions and the left-operand traffic per flop, and for two
// accumulator buffers (2 x 256 tensor-memory columns), so the epilogue of one tile runs under the
// main loop of the next.  A k-block is 128 BYTES of contraction per row for every operand type
// (64 bf16 or 128 codes), so all tiles are 128-byte-swizzled 16 KB blocks: a stage is this CTA's
// 128 left rows and its 128-row half of the right tile, 32 KB, five stages.  Roles, barriers,
// bounded waits and the exit protocol are those of tc_kernel.
constexpr int kWideN = 256;
constexpr int kWideHalfN = 128;
constexpr int kWideStages = 5;
constexpr uint32_t kWideTile = 128 * 128;                 // 16 KB
constexpr uint32_t kWideStageBytes = 2 * kWideTile;

struct SharedWide {
  uint64_t full[kWideStages];
  uint64_t empty[kWideStages];
  uint64_t tmem_full[2];         // per CTA, per accumulator buffer
  uint64_t tmem_empty[2];        // leader, per accumulator buffer
  uint32_t tmem_base;
  uint32_t abort_flag;
  float delta_r[2][kWideN];
  uint4 stage[kEpiWarps][32 * 8];  // output chunks on their way out, 4 KB per epilogue warp
};

// KIND: kKindF16 (bf16 x bf16 -> fp32 output), kKindF8 / kKindI8 (descaled and/or raw output)
template <int KIND>
__global__ void __launch_bounds__(kThreads, 1)
tc_gemm_wide_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                    const KernelArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  SharedWide* sh = reinterpret_cast<SharedWide*>(tiles + (size_t)kWideStages * kWideStageBytes);
  // known to the compiler to be the same in all lanes (see tc_group_kernel)
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;
  constexpr int kElemsPerBlock = KIND == kKindF16 ? 64 : 128;          // contraction elements per k-block
  const int num_kb = (int)((a.K + kElemsPerBlock - 1) / kElemsPerBlock);
  volatile uint32_t* abort_flag = &sh->abort_flag;

  if (warp == 0 && lane < 2) {
    const CUtensorMap* maps[2] = {&map_a, &map_b};
    asm volatile("prefetch.tensormap [%0];" ::"l"(maps[lane]) : "memory");
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < kWideStages; ++s) {
      mbar_init(smem_u32(&sh->full[s]), 1);
      mbar_init(smem_u32(&sh->empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&sh->tmem_full[b]), 1);
      mbar_init(smem_u32(&sh->tmem_empty[b]), 2 * kEpiWarps);
    }
    sh->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&sh->tmem_base)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  pdl_prologue();
  tc_fence_after();
  const uint32_t tmem_base = sh->tmem_base;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (both CTAs)
    if (lane == 0) {
      uint32_t g = 0;
      bool ok = true;
      for (int t = pair; t < a.num_tiles && ok; t += num_pairs) {
        const TileCoord tc = tile_coord(t, a);
        const int r0 = tc.m_tile * kPairM + (int)rank * kBlockM;
        const int c0 = tc.n_tile * kWideN + (int)rank * kWideHalfN;
        for (int kb = 0; kb < num_kb; ++kb, ++g) {
          const int s = g % kWideStages;
          const uint32_t use = g / kWideStages;
          if (use > 0 && !mbar_wait(smem_u32(&sh->empty[s]), (use - 1) & 1, abort_flag, a.err_word)) {
            ok = false;
            break;
          }
          if (rank == 0) mbar_expect_tx(smem_u32(&sh->full[s]), 2 * kWideStageBytes);
          const uint32_t bar = map_to_cta(smem_u32(&sh->full[s]), 0);
          const uint32_t base = smem_u32(tiles + (size_t)s * kWideStageBytes);
          tma_load_3d(base, &map_a, bar, kb * kElemsPerBlock, r0, tc.b);
          tma_load_3d(base + kWideTile, &map_b, bar, kb * kElemsPerBlock, c0, tc.b);
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (leader CTA, converged warp)
    if (rank == 0) {
      const bool lead = elect_one();
      const uint32_t idesc = KIND == kKindF16 ? make_idesc(1, 1, 1, kPairM, kWideN) : a.idesc_lp;
      uint32_t g = 0, it = 0;
      bool ok = true;
      for (int t = pair; t < a.num_tiles && ok; t += num_pairs, ++it) {
        const uint32_t buf = it & 1;
        // the buffer was last used by tile it-2: wait until both epilogues have drained it
        if (it >= 2 && !mbar_wait_warp(smem_u32(&sh->tmem_empty[buf]), ((it >> 1) - 1) & 1, abort_flag, a.err_word))
          break;
        tc_fence_after();
        for (int kb = 0; kb < num_kb; ++kb, ++g) {
          const int s = g % kWideStages;
          if (!mbar_wait_warp(smem_u32(&sh->full[s]), (g / kWideStages) & 1, abort_flag, a.err_word)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t base = smem_u32(tiles + (size_t)s * kWideStageBytes);
          const uint64_t da = smem_desc(base, 128), db = smem_desc(base + kWideTile, 128);
          if (lead) {
#pragma unroll
            for (int k = 0; k < 4; ++k)           // 32 bytes of contraction per instruction
              mma_pair<KIND>(tmem_base + buf * kWideN, da + 2 * k, db + 2 * k, idesc, k ? 1u : (uint32_t)kb, true);
            tc_commit_pair(smem_u32(&sh->empty[s]), true);
          }
        }
        if (ok) tc_commit_pair(smem_u32(&sh->tmem_full[buf]), lead);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue (warps 2..9, both CTAs)
    const int q = warp & 3;
    const int h = (warp - 2) >> 2;                // which 128-column half of the tile
    const int et = (warp - 2) * 32 + lane;        // 0..255
    const float dl_tensor = (KIND != kKindF16 && !a.pc_l) ? __ldg(a.dl) : 1.f;
    const float dr_tensor = (KIND != kKindF16 && !a.pc_r) ? __ldg(a.dr) : 1.f;
    const bool per_col = KIND != kKindF16 && a.pc_r;
    // 16-byte stores need 16-byte aligned rows: output bases aligned and N a multiple of 4
    const bool vec_ok = (a.N & 3) == 0 && (reinterpret_cast<uintptr_t>(a.out_descaled) & 15) == 0 &&
                        (reinterpret_cast<uintptr_t>(a.out_raw) & 15) == 0;
    uint4* const stage = sh->stage[warp - 2];
    uint32_t it = 0;
    for (int t = pair; t < a.num_tiles; t += num_pairs, ++it) {
      const TileCoord tc = tile_coord(t, a);
      const uint32_t buf = it & 1;
      float* dr_s = sh->delta_r[buf];
      if (per_col) {
        const int64_t col = (int64_t)tc.n_tile * kWideN + et;
        dr_s[et] = col < a.N ? __ldg(a.dr + (int64_t)tc.b * a.N + col) : 0.f;
      }
      const int64_t row0 = (int64_t)tc.m_tile * kPairM + rank * kBlockM + q * 32, row = row0 + lane;
      const bool row_ok = row < a.M;
      const int rows_live = (int)(a.M - row0 < 32 ? a.M - row0 : 32);      // <= 0: none
      float dlv = dl_tensor;
      if (KIND != kKindF16 && a.pc_l) dlv = row_ok ? __ldg(a.dl + (int64_t)tc.b * a.M + row) : 0.f;
      const bool ok = mbar_wait(smem_u32(&sh->tmem_full[buf]), (it >> 1) & 1, abort_flag, a.err_word);
      if (epi_barrier_any(!ok)) break;            // also publishes delta_r
      tc_fence_after();
      const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16) + buf * kWideN;
#pragma unroll 1
      for (int c = 0; c < 4; ++c) {
        const int cc0 = h * 128 + c * 32;
        const int64_t col0 = (int64_t)tc.n_tile * kWideN + cc0;
        if (col0 >= a.N) break;                   // uniform across the warp
        const int n_live = (int)(a.N - col0 < 32 ? a.N - col0 : 32);
        uint32_t r[32];
        tmem_ld32(lane_addr + cc0, r);
        tmem_ld_wait();
        const int64_t o0 = ((int64_t)tc.b * a.M + row0) * a.N + col0;     // first row of the warp, first column of the chunk
        if (KIND == kKindF16) {
          store_chunk(stage, lane, r, reinterpret_cast<uint32_t*>(a.out_descaled) + o0, a.N, rows_live, n_live, vec_ok);
        } else {
          if (a.out_raw) store_chunk(stage, lane, r, reinterpret_cast<uint32_t*>(a.out_raw) + o0, a.N, rows_live, n_live, vec_ok);
          if (a.out_descaled) {
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              const float acc = KIND == kKindI8 ? (float)(int)r[j] : __uint_as_float(r[j]);
              r[j] = __float_as_uint(acc * (dlv * (per_col ? dr_s[cc0 + j] : dr_tensor)));
            }
            store_chunk(stage, lane, r, reinterpret_cast<uint32_t*>(a.out_descaled) + o0, a.N, rows_live, n_live, vec_ok);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(map_to_cta(smem_u32(&sh->tmem_empty[buf]), 0));
    }
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

// ------------------------------------------------------------------ the fused probe kernel
// One persistent launch computes the Eq. 3 records of many probes.  Probes of the same two operands
// (a sweep of formats or granularities over one product) share the reference L.R and the
// denominator |L|.|R|, which do not depend on the format, so they form one UNIT: per output tile the
// reference and denominator products run once, then the 8-bit products of the unit's probes
// (VARIANTS, up to kMaxVar) one after the other, each over the whole contraction.
//
// The host orders the units by descending tile cost and deals the tiles of each to the CTA pairs with the least
// to do so far (TileDeal); the deal is fixed, so that records are the same from run to run.  The operand maps, scales, shapes and the 8-bit MMA kinds come
// from a table in the kernel's parameter space.  A pair meets each unit in
// one run: when the unit changes, the epilogue warps reduce their statistics and write the CTA's
// records of the probes they leave.
//
// What bounds this kernel is shared-memory bandwidth, about 128 B per clock and SM for TMA writes, MMA
// operand reads and ordinary accesses together, and under sustained load the power limit.  Per 64
// contraction entries of a 256 x 128 tile the reference and denominator products move 72 KB (24 KB
// by TMA, 16 KB of MMA operands, 32 KB by the converters; 512 tensor cycles) and an 8-bit product 24 KB
// (12 + 12; 128 tensor cycles).  A product in F formats so costs 72 + 24 F KB per k-block against F
// times 112 for separate probes with all three products side by side.  Measured (16384 x 4096 x 1024,
// fused kernel only, same GPU): one format 284 us (separate 282), three 420 (793), six 660 (1624).
// Running the products one after the other, instead of side by side on narrower tiles, is what keeps
// the tiles 128 wide: five accumulators side by side would leave room for 64 columns each, at 256 KB
// per 128 columns against the 144 KB here.  (Units of one probe have nothing to share: tc_side_kernel.)
//
// The left operand of the reference and denominator products is not read from shared memory by the tensor
// cores: converter warps read this CTA's 128 rows of the L tile once and store them, and the same with
// the sign bits cleared, into TENSOR memory, from where both products take their A operand; two more warps, or where
// contractions are short the converters too (r_by_warps), write the |R| half-tile into the stage.  No |x| copy exists in HBM.  What the bf16 phase waits for is the
// converters' serial time per block: wait, loads, wait for the tensor-memory stage, stores, arrival (4096^2 x 1024 in three
// formats, cycles per block: 760 with |R| among the converters' work, 683 with two warps for it; 553 with all conversions left
// out; four stages in tensor memory instead of two change nothing).  Half-block stages and prefetching the next
// block's values ahead of the fences each measured 5 to 20 % slower.
//
// Operands whose contraction is strided are staged as they lie in memory (mn-major tiles, a contraction entry per 128-byte
// row): the tensor cores read R and the codes so at the rate of contraction-major ones, the converters turn L with
// ldmatrix.  No copy of an operand is made, and under one scale a tensor that is used in both orientations is quantized
// once, in its own order.  8192 x 4096 x 1024 in three formats, both operands contiguous / strided: 217 / 213 us.
//
// Roles in each CTA (512 threads = 4 warpgroups; registers are re-divided with setmaxnreg):
//   warp 0        TMA producer: blocks of the ring of kStages stages in the order of consumption: per tile
//                 the k-blocks of L and R (64 entries deep), then per variant those of its codes
//                 (128 deep); both kinds bring 128 bytes per row.  A CTA's loads complete on its own `full`.
//   warp 1        allocates tensor memory; in the leader CTA it runs the MMA loop converged and
//                 one elected lane issues the pair's MMAs; tcgen05.commit frees a stage in both CTAs (`empty`).
//   warps 2, 3    |R|: a sign-cleared copy of each staged R half-tile (idle where the converters write it).
//   warps 4..7    converters of L, one per tensor-memory lane quarter: thread = one of the CTA's 128
//                 left-operand rows.  Blocks of codes need no conversion: they only pass on that they landed.
//   warps 8..15   epilogue.
// Tensor memory: columns 0..127 reference, 128..255 denominator, 256..383 and 384..511 two 8-bit
// accumulators.  The second one doubles as two stages of L and |L| (32 columns of two bf16 each): it
// is only written between a tile's denominator product and the next tile's, because variant f of F uses
// accumulator (F-1-f) & 1, so that the last variant of a tile never needs it and the next tile's
// converters start under the last variant's MMAs.
//   The epilogue copies its reference and denominator columns into registers when they are complete
// (`rd_full`) and hands both blocks back at once (`rd_empty`); while the first 8-bit product runs it
// forms the sums of C^2 and D^2 and replaces D by its reciprocal, so that evaluating a variant costs
// 3 to 4 instructions per output.  The 8-bit accumulators come and go through `lp_full` / `lp_done`, one
// pair of barriers each; `abs_free` tells this CTA's converters that the second one has been read.  No
// M x N matrix ever goes to HBM.
constexpr int kMaxVar = 6;                     // probes of one unit (three formats at two granularities)
constexpr int kProbeThreads = 512;
constexpr int kFirstEpiWarp = 8;               // warps 8..15: lane quarter = warp % 4 holds for both groups
// registers per thread after the split (launch: 128 each): 72 + 88 + 176 + 176 = 4 x 128
constexpr int kRegsCtl = 72, kRegsConv = 88, kRegsEpi = 176;
static_assert(kRegsCtl + kRegsConv + 2 * kRegsEpi <= 4 * 128, "the split must fit what the block was launched with");

struct CfgP {
  static constexpr int kStages = 6;          // stages of shared memory (TMA ring)
  static constexpr int kTmemStages = 2;       // stages of L and |L| in tensor memory (128 columns / 64)
  static constexpr int kLpDepth = 128;       // contraction entries of a block of codes
  // stage: L, R, |R| (written by warps 2 and 3 or the converters); or codes of L, codes of R.  All rows are 128 bytes.
  static constexpr uint32_t kOffL = 0, kOffR = kABf16, kOffRa = kOffR + kBBf16;
  static constexpr uint32_t kStageBytes = kOffRa + kBBf16;           // 32 KB
  static constexpr uint32_t kTileBytes = kStages * kStageBytes;      // 192 KB
  static constexpr uint32_t kColRef = 0, kColDen = 128, kColLp = 256, kColL = 384;   // tensor-memory columns
};

// Division of a tile's position (below 2^31) by a number of tiles without a divide instruction: with 2^(s-1) < d <= 2^s and
// mul = floor(2^(31+s) / d) + 1 the quotient of n is the upper half of 2 n mul, shifted right by s (the excess of mul adds less
// than 1 / d for such n).
struct Divisor {
  uint32_t mul, shift;
  __host__ explicit Divisor(uint32_t d) : shift(0) {
    while ((1ull << shift) < d) ++shift;
    mul = (uint32_t)((1ull << (31 + shift)) / d + 1);
  }
};
__device__ __forceinline__ uint32_t divide(uint32_t n, uint32_t mul, uint32_t shift) { return __umulhi(n << 1, mul) >> shift; }

// What the roles need of a unit for every tile, copied to shared memory once per CTA: the
// launch's table sits in the kernel's parameter space, and reads of it with an index known only
// at run time go through the small constant cache, which a table of this size thrashes.
struct alignas(16) WalkInfo {
  int32_t n_tiles, n_lead, lead0, main0;            // this pair's tiles of the unit: lead0 + j for its j-th tile while
                                                    // j < n_lead, then main0 + j * pairs, the last one `last` unless -1
  int32_t per_b, inner, num_kb, half_n;             // per_b = tiles_m * tiles_n (tiles per batch element);
                                                    // inner = tiles_n: column tiles run fastest, -tiles_m: row tiles do;
                                                    // half_n: kUnitMnMajor... above its low byte, the unit's index above those
  uint32_t b_mul, b_shift, i_mul, i_shift;          // division by per_b and by the absolute value of inner (Divisor)
  int32_t n_var, var_begin, K, last;
};
// Of a probe: the instruction descriptor of its 8-bit MMA, and kVar...; per-channel scales are indexed by batch * M + row,
// batch * N + column.
struct VarInfo { uint32_t idesc, flags; };
enum : uint32_t { kVarI8 = 1, kVarScalePerRow = 2, kVarScalePerCol = 4, kVarRowStats = 8, kVarMnMajorL = 16, kVarMnMajorR = 32 };
enum : uint32_t { kUnitMnMajorL = 1, kUnitMnMajorR = 2 };

template <int UNITS, int VARS>
struct SharedP {
  uint64_t full[CfgP::kStages];     // per CTA: this CTA's loads of a block have landed
  uint64_t ready[CfgP::kStages];    // leader: both CTAs' converters (and warps 2 and 3, with RW) have seen their loads
                                    //         land and, for L and R, have written L and |L| (tensor memory) and |R| (stage)
  uint64_t empty[CfgP::kStages];    // per CTA: the pair's MMAs have finished with the block of the stage
  uint64_t rd_full;                 // per CTA: the tile's reference and denominator are complete
  uint64_t rd_empty;                // leader: both CTAs' epilogues have copied them out
  uint64_t lp_full[2];              // per CTA: an 8-bit accumulator is complete
  uint64_t lp_done[2];              // leader: both CTAs' epilogues have read it
  uint64_t abs_free;                // per CTA: this CTA's epilogue has read the tile's last use of the second 8-bit accumulator
  uint64_t drain;                   // leader, give-up path only: every MMA issued so far has completed
  uint32_t tmem_base;
  uint32_t abort_flag;
  uint32_t is_last;
  uint32_t issued;                  // blocks whose loads the producer has issued (read on the give-up path)
  float delta_r[2][kMaxVar][kBlockN];
  // per warp and pair of rows (lanes l and l + 16): sum BE, sum diff^2, max BE of each variant of the unit
  double2 sums[kMaxVar][kEpiWarps][16];
  float maxima[kMaxVar][kEpiWarps][16];
  double red[3 * kMaxVar + 2][kEpiWarps];
  float dl_tensor[kMaxVar], dr_tensor[kMaxVar];     // per-tensor scales of the unit in hand (1 where per channel)
  int32_t n_walk;                   // units that give this pair tiles
  WalkInfo walk[UNITS];
  VarInfo var[VARS];
};

constexpr int kMaxPairs = 80;               // CTA pairs of a launch, at most (148 SMs hold 74)
// (A unit's words are one line of the constant cache, and so are a probe's: every line is a miss of its own at the start of a launch, which
// takes 600 cycles of a launch of eight units.)
struct alignas(64) GroupUnit {
  int32_t M, N, K;
  int32_t tiles_m, tiles_n;
  int32_t rounds;             // tiles that every pair takes of it, after those of GroupTable::lead
  int32_t n_lead;             // of all pairs together, those of GroupTable::lead
  int32_t half_n;             // right-operand rows each CTA stages: 64, or 32 for outputs at most 64 wide
  uint32_t last[(kMaxPairs + 31) / 32];   // bit p: pair p takes one more after them
  uint32_t major;             // kUnitMnMajor...: bf16 operands stored with the contraction strided
  uint32_t b_mul, i_mul;      // see WalkInfo
  uint8_t b_shift, i_shift;
  uint8_t m_fastest;          // the tiles of a batch element are walked down the rows first (below)
  int16_t var_begin, n_var;
};
static_assert(sizeof(GroupUnit) == 64, "a line");
struct alignas(64) GroupVar {
  const float* dl; const float* dr;
  double* partials;           // gridDim.x records
  double* row_stats;          // optional [batch * M][5] per-row sums
  qm_metric_result* result;
  uint32_t* err_word;
  const uint32_t* err_also[2];           // further error words to report in the record, or null
};
static_assert(sizeof(GroupVar) == 64, "a line");
template <int UNITS, int VARS>
struct GroupTable {
  static constexpr int kUnits = UNITS, kVars = VARS;
  static_assert(VARS <= 64, "a bit to a probe");
  CUtensorMap unit_maps[UNITS][2];        // L, R
  CUtensorMap var_maps[VARS][2];          // codes of L, codes of R
  int32_t n, n_var;
  uint32_t stop_after_kb;     // test hook: the producer issues no block beyond this many (0xffffffff: off)
  uint64_t wait_limit_ns;     // bound of every barrier wait
  uint32_t* done_counter;     // zero on entry; counts finished CTAs
  uint32_t* err0;             // a wait that runs out is reported here and in every record
  const uint32_t* prepare_flags;          // of a single probe: flag words of the operands' preparation, or null
  GroupUnit u[UNITS];
  GroupVar v[VARS];
  VarInfo info[VARS];
  uint64_t count[VARS];                   // batch * M * N
  uint8_t first[kMaxPairs];               // the first unit that gives a pair tiles
  uint16_t lead[UNITS][kMaxPairs + 1];    // prefix sums over the pairs of the tiles that each takes ahead of the unit's rounds
};
// A launch's table has to fit into 32 764 bytes of kernel parameters.  24 units hold the 18 products
// of an encoder layer in one launch; a probe on its own passes a table of its own size (1 KB).
using TableBig = GroupTable<24, 56>;
using TableOne = GroupTable<1, 1>;
static_assert(sizeof(TableBig) <= 32764, "kernel parameters");

// What a unit asks of every role, read once per unit: the same in all lanes, and known to be (the shuffles).  A tile's own
// code is kept short by this: 512 x 512 x 64 x 256 in one format 95 us with one loop over tiles that looks its unit up, 87 so.
// The roles go through the units that give their pair tiles and no others: going past the rest took 18 small products 3 us of 31.
struct UnitInfo {
  int unit, n_tiles, num_kb, half_n, n_var, var_begin, K;
  uint32_t major;
  __device__ __forceinline__ explicit UnitInfo(const WalkInfo& w) {
    constexpr uint32_t all = 0xffffffffu;
    n_tiles = __shfl_sync(all, w.n_tiles, 0);
    num_kb = __shfl_sync(all, w.num_kb, 0);
    const int h = __shfl_sync(all, w.half_n, 0);
    half_n = h & 255; major = (uint32_t)h >> 8 & 255u; unit = h >> 16;
    n_var = __shfl_sync(all, w.n_var, 0);
    var_begin = __shfl_sync(all, w.var_begin, 0);
    K = __shfl_sync(all, w.K, 0);
  }
  __device__ __forceinline__ int lp_blocks() const { return (K + CfgP::kLpDepth - 1) / CfgP::kLpDepth; }
};
// The pair's j-th tile of a unit.  Every role goes through the units and their tiles in the same order; the producer
// and the epilogue also need to know where the tiles are.
__device__ __forceinline__ TileCoord pair_tile(const WalkInfo& w, int j, int num_pairs) {
  const int4 s4 = reinterpret_cast<const int4*>(&w)[0];        // n_tiles, n_lead, lead0, main0
  const int4 w4 = reinterpret_cast<const int4*>(&w)[1];        // per_b, inner, num_kb, half_n
  const uint4 d4 = reinterpret_cast<const uint4*>(&w)[2];
  const uint32_t t = (uint32_t)(j + 1 == s4.x && w.last >= 0 ? w.last : j < s4.y ? s4.z + j : s4.w + j * num_pairs);
  const uint32_t b = divide(t, d4.x, d4.y);
  const uint32_t rem = t - b * (uint32_t)w4.x;
  const int inner = w4.y < 0 ? -w4.y : w4.y;
  const int outer_i = (int)divide(rem, d4.z, d4.w), inner_i = (int)rem - outer_i * inner;
  TileCoord tc;
  tc.b = (int)b;
  tc.m_tile = w4.y < 0 ? inner_i : outer_i;
  tc.n_tile = w4.y < 0 ? outer_i : inner_i;
  return tc;
}

// Position in a ring of stages.
template <int STAGES>
struct Ring {
  uint32_t s = 0, parity = 0;       // stage, and the parity of its use
  __device__ __forceinline__ void next() {
    if (++s == (uint32_t)STAGES) { s = 0; parity ^= 1u; }
  }
};

// Bounded wait with the launch's limit; see mbar_wait.
struct Waiter {
  volatile uint32_t* abort_flag;
  uint32_t* err_word;
  uint64_t limit_ns;
  __device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity) const {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = global_timer_ns();
    uint32_t polls = 0;
    while (true) {
      if (mbar_try_wait(bar, parity)) return true;
      if ((++polls & 0x3fu) == 0) {
        if (*abort_flag) return false;
        if (global_timer_ns() - t0 > limit_ns) {
          *abort_flag = 1u;
          if (err_word) atomicOr(err_word, QM_DEVERR_TIMEOUT);
          return false;
        }
      }
    }
  }
  __device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity) const {
    return __all_sync(0xffffffffu, wait(bar, parity));
  }
};

// Tile load into this CTA's shared memory, completing on this CTA's barrier.
__device__ __forceinline__ void tma_load_3d_local(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1,
                                                  int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts128(uint32_t addr, uint4 v) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
// 32 lanes x 32 consecutive 32-bit columns of tensor memory from registers: lane (base + t) <- thread t.
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
        "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
        "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
// 16 lanes x 32 consecutive 32-bit columns: thread t holds words 4 n + t % 4 of row t / 4 in r[2 n] and of row 8 + t / 4 in
// r[2 n + 1], which is how ldmatrix leaves 8 x 8 matrices.
__device__ __forceinline__ void tmem_st16x32(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x128b.x8.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
// Four transposed 8 x 8 matrices of 16-bit values; lane l gives the address of row l % 8 of matrix l / 8.
__device__ __forceinline__ void ldmatrix4_trans(uint32_t addr, uint32_t* r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// A mn-major L tile (64 contraction entries x 128 operand rows, as two 128-byte-swizzled boxes of 64 rows) for the 32 rows of
// lane quarter q: a[16 h + ...] holds rows 16 h .. 16 h + 15 in the form of tmem_st16x32.  A matrix is 8 entries x 8 rows, its
// eight 16-byte pieces on different banks by the swizzle.
__device__ __forceinline__ void load_l_mn_major(uint32_t base, int q, int lane, uint32_t (&a)[32]) {
  const uint32_t rr = (uint32_t)lane & 7u, mi = (uint32_t)lane >> 3;
  const uint32_t box = base + (uint32_t)(q >> 1) * 8192u + (8u * (mi >> 1) + rr) * 128u;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t at = box + ((((uint32_t)(q & 1) * 4u + (uint32_t)h * 2u + (mi & 1u)) ^ rr) << 4);
#pragma unroll
    for (int n = 0; n < 4; ++n) ldmatrix4_trans(at + (uint32_t)n * 2048u, &a[16 * h + 4 * n]);
  }
}
// |R| beside a staged R half-tile, whatever its order: a flat sign-cleared copy of its first `vectors` 16-byte vectors (at most
// 512) by the THREADS threads t = 0 .. THREADS - 1.  The tensor core sees it after a fence.proxy.async.
template <int THREADS>
__device__ __forceinline__ void abs_r(uint32_t r, uint32_t to_abs, int vectors, int t) {
  constexpr int kEach = 512 / THREADS;
  const uint32_t src = r + (uint32_t)t * 16u, m = 0x7fff7fffu;
  uint4 u[kEach];
#pragma unroll
  for (int j = 0; j < kEach; ++j) u[j] = t + THREADS * j < vectors ? lds128(src + (uint32_t)j * (16u * THREADS)) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
  for (int j = 0; j < kEach; ++j)
    if (t + THREADS * j < vectors)
      sts128(src + to_abs + (uint32_t)j * (16u * THREADS), make_uint4(u[j].x & m, u[j].y & m, u[j].z & m, u[j].w & m));
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// 32 lanes x 8 consecutive 32-bit columns.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(taddr)
      : "memory");
}
// D[256 x N] (+)= A[256 x 16] . B[N x 16]^T across the CTA pair, A (bf16) taken from tensor memory:
// each CTA's 128 rows at the same column address, two values per 32-bit column.
__device__ __forceinline__ void mma_pair_a_tmem(uint32_t tmem_d, uint32_t tmem_a, uint64_t db, uint32_t idesc,
                                                uint32_t accumulate, bool lead) {
  if (!lead) return;
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(tmem_d), "r"(tmem_a), "l"(db), "r"(idesc), "r"(accumulate) : "memory");
}

// Eq. 3 statistics of one row of one variant's tile.
struct StatsV {
  float be0, be1, mx;
  uint64_t d2;
};
// Eight consecutive columns of a row: reference rc, reciprocal denominator ri, raw 8-bit accumulator rq.
// PER_COL: the right operand has a scale per column (dr_s) and kd2 holds -delta_l twice, otherwise
// kd2 holds (-delta_l delta_r) twice.
template <bool PER_COL>
__device__ __forceinline__ void eval8(const uint32_t* rc, const uint32_t* ri, uint32_t (&rq)[8], bool is_i8, uint64_t kd2,
                                      const float* dr_s, StatsV& s) {
  if (is_i8) {
#pragma unroll
    for (int j = 0; j < 8; ++j) rq[j] = __float_as_uint((float)(int)rq[j]);
  }
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    const uint64_t a2 = pack2(__uint_as_float(rq[j]), __uint_as_float(rq[j + 1]));
    const uint64_t cv2 = pack2(__uint_as_float(rc[j]), __uint_as_float(rc[j + 1]));
    uint64_t diff2;                                              // C - A dl dr
    if (PER_COL) diff2 = fma2(mul2(a2, kd2), *reinterpret_cast<const uint64_t*>(dr_s + j), cv2);
    else diff2 = fma2(a2, kd2, cv2);
    const uint64_t be2 = mul2(diff2, pack2(__uint_as_float(ri[j]), __uint_as_float(ri[j + 1])));
    float b0, b1;
    unpack2(be2, b0, b1);
    s.be0 += fabsf(b0);
    s.be1 += fabsf(b1);
    s.mx = fmaxf(s.mx, fmaxf(fabsf(b0), fabsf(b1)));
    s.d2 = fma2(diff2, diff2, s.d2);
  }
}
// One variant of a tile for this warp's lane quarter and columns: the accumulator comes eight columns at
// a time, the next eight on their way while eight are evaluated; `release` runs (converged) as soon as
// the last ones are in registers.  live = columns of this warp that exist in the matrix (may be <= 0).
template <bool PER_COL, typename Release>
__device__ __forceinline__ void eval_variant(uint32_t taddr, const uint32_t (&rc)[64], const uint32_t (&ri)[64], int live,
                                             bool is_i8, uint64_t kd2, const float* dr_s, StatsV& st, Release release) {
  uint32_t q0[8], q1[8];
  if (live <= 0) { release(); return; }
  tmem_ld8(taddr, q0);
  tmem_ld_wait();
#pragma unroll
  for (int p = 0; p < 4; ++p) {                    // 16 columns per step
    if (p * 16 >= live) break;
    const bool more = p < 3 && (p + 1) * 16 < live;
    tmem_ld8(taddr + p * 16 + 8, q1);
    eval8<PER_COL>(&rc[p * 16], &ri[p * 16], q0, is_i8, kd2, dr_s + p * 16, st);
    tmem_ld_wait();
    if (more) tmem_ld8(taddr + p * 16 + 16, q0);
    else release();
    eval8<PER_COL>(&rc[p * 16 + 8], &ri[p * 16 + 8], q1, is_i8, kd2, dr_s + p * 16 + 8, st);
    if (more) tmem_ld_wait();
  }
}

// The operand maps of the pair's first tile into the descriptor cache (one warp).
template <typename Table>
__device__ __forceinline__ void prefetch_maps(const Table& tab, int lane, int pair) {
  if (lane < 4) {
    const int pi = Table::kUnits > 1 ? tab.first[pair] : 0;
    const CUtensorMap* m = lane < 2 ? &tab.unit_maps[pi][lane] : &tab.var_maps[tab.u[pi].var_begin][lane - 2];
    asm volatile("prefetch.tensormap [%0];" ::"l"(m) : "memory");
  }
}
// The walk of this pair (the units that give it tiles, in order) and the variant table of a launch into shared memory (one warp).
template <typename Sh, typename Table>
__device__ __forceinline__ void fill_walk(Sh* sh, const Table& tab, int lane, int pair, int num_pairs) {
  static_assert(Table::kUnits <= 32, "a lane to a unit");
  WalkInfo wi;
  wi.n_tiles = 0;
  const GroupUnit& u = tab.u[lane < tab.n ? lane : 0];
  if (lane < tab.n) {
    const int32_t rounds = u.rounds, n_lead = u.n_lead;
    const uint32_t last0 = u.last[0], last1 = u.last[1], last2 = u.last[2];
    const int32_t tiles_m = u.tiles_m, tiles_n = u.tiles_n;
    wi.K = u.K; wi.b_mul = u.b_mul; wi.i_mul = u.i_mul; wi.b_shift = u.b_shift; wi.i_shift = u.i_shift;
    wi.n_var = u.n_var; wi.var_begin = u.var_begin;
    wi.half_n = u.half_n | (int32_t)(u.major << 8) | lane << 16;
    wi.inner = u.m_fastest ? -tiles_m : tiles_n;
    wi.per_b = tiles_m * tiles_n;
    wi.num_kb = (wi.K + kBlockK - 1) / kBlockK;
    wi.lead0 = wi.n_lead = 0;
    if (n_lead > 0) {                                // (rows of their own in the table, seldom needed)
      wi.lead0 = tab.lead[lane][pair];
      wi.n_lead = tab.lead[lane][pair + 1] - wi.lead0;
    }
    wi.n_tiles = wi.n_lead + rounds;
    wi.main0 = n_lead + pair - wi.n_lead * num_pairs;
    const uint32_t below = (1u << (pair & 31)) - 1u, word = pair < 32 ? last0 : pair < 64 ? last1 : last2;
    wi.last = -1;
    if (word >> (pair & 31) & 1u) {
      wi.last = n_lead + rounds * num_pairs + __popc(word & below) + (pair >= 32 ? __popc(last0) : 0) + (pair >= 64 ? __popc(last1) : 0);
      ++wi.n_tiles;
    }
  }
  const uint32_t mine = __ballot_sync(0xffffffffu, wi.n_tiles > 0);
  if (wi.n_tiles > 0) sh->walk[__popc(mine & ((1u << lane) - 1u))] = wi;
  if (lane == 0) sh->n_walk = __popc(mine);
  for (int i = lane; i < tab.n_var; i += 32) sh->var[i] = tab.info[i];
}

// Sums of four values over the warp, six exchanges instead of twenty: lanes 8 k .. 8 k + 7 return the sum of v[k].
__device__ __forceinline__ double warp_sum4(double v0, double v1, double v2, double v3, int lane) {
  const bool hi = lane & 16, odd = lane & 8;
  double a = hi ? v2 : v0, b = hi ? v3 : v1;
  a += __shfl_xor_sync(0xffffffffu, hi ? v0 : v2, 16);
  b += __shfl_xor_sync(0xffffffffu, hi ? v1 : v3, 16);
  double x = odd ? b : a;
  x += __shfl_xor_sync(0xffffffffu, odd ? a : b, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
// Maximum of values that are not negative (nor NaN).
__device__ __forceinline__ float warp_max_f(float x) { return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(x))); }

// Every record of the launch is visible (last CTA): epilogue warp ew takes probes ew, ew + 8, ...; fixed-order
// sum (lane l takes records l, l + 32, ...).  One round trip to L2 per probe: 4 200 cycles with a trip for each 32
// records and one per flag word.
template <typename Table>
__device__ __forceinline__ void write_results(const Table& tab, int ew, int lane) {
  constexpr int kTake = 5;                           // records of a lane on their way together: 160 in a warp
  for (int vi = ew; vi < tab.n_var; vi += kEpiWarps) {
    const GroupVar& a = tab.v[vi];
    // four lanes fetch the words that make up the record's flags
    const uint32_t* word = lane == 0 ? a.err_word : lane == 1 ? a.err_also[0] : lane == 2 ? a.err_also[1] : lane == 3 ? tab.err0 : nullptr;
    uint32_t flags = word ? *reinterpret_cast<const volatile uint32_t*>(word) : 0u;
    if (lane == 3) flags &= QM_DEVERR_TIMEOUT;
    if (Table::kUnits == 1 && tab.prepare_flags) {
      uint32_t any = 0;
#pragma unroll
      for (int i = 0; i < kPrepareFlagWords; i += 32)
        if (i + lane < kPrepareFlagWords) any |= __ldcg(tab.prepare_flags + i + lane);
      if (any) flags |= QM_DEVERR_NONFINITE;
    }
    double s4[4] = {0, 0, 0, 0};
    float mx = 0.f;
    for (int i0 = lane; i0 < (int)gridDim.x; i0 += 32 * kTake) {
      double r[kTake][kPartialDoubles];
#pragma unroll
      for (int u = 0; u < kTake; ++u) {
        const int i = i0 + 32 * u;
        const double* rec = a.partials + (int64_t)i * kPartialDoubles;
#pragma unroll
        for (int k = 0; k < kPartialDoubles; ++k) r[u][k] = i < (int)gridDim.x ? __ldcg(rec + k) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < kTake; ++u) {
        s4[0] += r[u][0]; s4[1] += r[u][2]; s4[2] += r[u][3]; s4[3] += r[u][4];
        mx = fmaxf(mx, (float)r[u][1]);              // (a float that was widened)
      }
    }
    const double x = warp_sum4(s4[0], s4[1], s4[2], s4[3], lane);
    mx = warp_max_f(mx);
    flags = __reduce_or_sync(0xffffffffu, flags);
    if (lane == 0) {                         // (the record may be in host memory: stores only, every field once)
      a.result->sum_be = x; a.result->max_be = (double)mx;
      a.result->count = tab.count[vi]; a.result->device_error = flags; a.result->reserved = 0;
    } else if (lane == 8) {
      a.result->sum_diff2 = x;
    } else if (lane == 16) {
      a.result->sum_ref2 = x;
    } else if (lane == 24) {
      a.result->sum_den2 = x;
    }
  }
}

// Common exit.  Neither CTA may leave while the other can still read its shared memory, signal its barriers
// or write its tensor memory, and no bulk load may still be writing into a CTA that retires.
template <int STAGES, typename Sh>
__device__ __forceinline__ void probe_exit(Sh* sh, uint64_t wait_limit_ns, int warp, uint32_t rank, uint32_t tmem_base) {
  tc_fence_before();
  __syncthreads();
  if (sh->abort_flag && threadIdx.x == 0) {
    // give-up path: the loads of the last STAGES blocks this producer issued may not have been
    // awaited by anyone; wait (bounded) until each has landed
    const uint32_t n = sh->issued;
    for (uint32_t j = n > (uint32_t)STAGES ? n - STAGES : 0u; j < n; ++j) {
      const uint32_t bar = smem_u32(&sh->full[j % STAGES]), parity = (j / STAGES) & 1;
      const uint64_t t0 = global_timer_ns();
      while (!mbar_try_wait(bar, parity) && global_timer_ns() - t0 < wait_limit_ns) {}
    }
  }
  if (sh->abort_flag && warp == 1 && rank == 0) {
    // ... and the MMAs issued so far may still be running: one more commit, awaited (bounded) here
    __syncwarp();
    if (elect_one())
      asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                       smem_u32(&sh->drain)) : "memory");
    __syncwarp();
    const uint64_t t0 = global_timer_ns();
    while (!mbar_try_wait(smem_u32(&sh->drain), 0) && global_timer_ns() - t0 < wait_limit_ns) {}
    __syncwarp();
  }
  __syncthreads();
  cluster_sync();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

// MN: units may have operands whose contraction is strided.  RW: |R| by warps of its own, not by the converters (r_by_warps).
template <typename Table, bool MN, bool RW>
__global__ void __launch_bounds__(kProbeThreads, 1)
tc_group_kernel(const __grid_constant__ Table tab) {
  using C = CfgP;
  using Sh = SharedP<Table::kUnits, Table::kVars>;
  constexpr int kStages = C::kStages, kTmemStages = C::kTmemStages;
  extern __shared__ uint8_t smem_raw[];
  // tiles start on a 1024-byte boundary (the 128-byte swizzle atom); the offset is the same in
  // both CTAs of the pair because their dynamic shared memory starts at the same address
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  Sh* sh = reinterpret_cast<Sh*>(tiles + C::kTileBytes);
  const uint32_t tile_base = smem_u32(tiles);

  // the shuffle tells the compiler that the warp index, and with it every role's control flow, is the same in all
  // lanes: four MMAs and a commit took the MMA warp 690 cycles to issue without it, a 128-deep block of codes 841; 477 so
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;
  const Waiter w{&sh->abort_flag, tab.err0, tab.wait_limit_ns};

  if (warp == 0) prefetch_maps(tab, lane, pair);
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&sh->full[s]), 1);
      mbar_init(smem_u32(&sh->ready[s]), 2 * (RW ? 6 : 4));   // four converter warps and, with RW, two for |R| in each CTA
      mbar_init(smem_u32(&sh->empty[s]), 1);
    }
    mbar_init(smem_u32(&sh->rd_full), 1);
    mbar_init(smem_u32(&sh->rd_empty), 2 * kEpiWarps);
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&sh->lp_full[b]), 1);
      mbar_init(smem_u32(&sh->lp_done[b]), 2 * kEpiWarps);
    }
    mbar_init(smem_u32(&sh->abs_free), kEpiWarps);
    mbar_init(smem_u32(&sh->drain), 1);
    sh->abort_flag = 0;
    sh->is_last = 0;
    sh->issued = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&sh->tmem_base)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  if (warp == 2) fill_walk(sh, tab, lane, pair, num_pairs);
  tc_fence_before();
  __syncthreads();
  cluster_arrive();
  tc_fence_after();
  const uint32_t tmem_base = sh->tmem_base;
  auto begin = [&]() {
    cluster_wait();        // the peer's barriers and tensor memory exist before anyone uses them
    pdl_prologue();        // everything above overlapped the tail of the previous kernel
    tc_fence_after();
  };

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsCtl));
    if (warp == 0) {
      // ---------------------------------------------------------- TMA producer (both CTAs)
      begin();
      if (lane == 0) {
        Ring<kStages> ring;
        uint32_t g = 0;
        bool ok = true;
        // a mn-major tile has the operand's rows as its inner coordinate; of bf16, 128 of them are two boxes
        auto load = [&](const CUtensorMap* maps, uint32_t bytes, int k0, int r0, int c0, int b, bool l_mn, bool r_mn, bool two_boxes) {
          // test hook: the consumers' waits run out
          if (g >= tab.stop_after_kb || (g >= (uint32_t)kStages && !w.wait(smem_u32(&sh->empty[ring.s]), ring.parity ^ 1u))) {
            ok = false;
            return;
          }
          const uint32_t bar = smem_u32(&sh->full[ring.s]), base = tile_base + ring.s * C::kStageBytes;
          mbar_expect_tx(bar, bytes);
          tma_load_3d_local(base + C::kOffR, &maps[1], bar, r_mn ? c0 : k0, r_mn ? k0 : c0, b);
          tma_load_3d_local(base + C::kOffL, &maps[0], bar, l_mn ? r0 : k0, l_mn ? k0 : r0, b);
          if (two_boxes) tma_load_3d_local(base + C::kOffL + kABf16 / 2, &maps[0], bar, r0 + 64, k0, b);
          sh->issued = ++g;
          ring.next();
        };
        for (int k = 0; k < sh->n_walk && ok; ++k) {
          const WalkInfo& wk = sh->walk[k];
          const int pi = wk.half_n >> 16;
          const int n_tiles = wk.n_tiles, num_kb = wk.num_kb, half_n = wk.half_n & 255, n_var = wk.n_var, v0 = wk.var_begin;
          const uint32_t major = (uint32_t)wk.half_n >> 8 & 255u;
          const int nb = (wk.K + C::kLpDepth - 1) / C::kLpDepth;
          const uint32_t bytes = kABf16 + (uint32_t)half_n * 128u;
          const bool l_mn = MN && (major & kUnitMnMajorL), r_mn = MN && (major & kUnitMnMajorR);
          for (int j = 0; j < n_tiles && ok; ++j) {
            const TileCoord tc = pair_tile(wk, j, num_pairs);
            const int r0 = tc.m_tile * kPairM + (int)rank * kBlockM;     // this CTA's left-operand rows
            const int c0 = tc.n_tile * kBlockN + (int)rank * half_n;     // this CTA's half of the right operand
            for (int kb = 0; kb < num_kb && ok; ++kb)
              load(tab.unit_maps[pi], bytes, kb * kBlockK, r0, c0, tc.b, l_mn, r_mn, l_mn);
            for (int f = 0; f < n_var && ok; ++f) {
              const uint32_t flags = sh->var[v0 + f].flags;
              for (int kb = 0; kb < nb && ok; ++kb)
                load(tab.var_maps[v0 + f], bytes, kb * C::kLpDepth, r0, c0, tc.b, MN && (flags & kVarMnMajorL), MN && (flags & kVarMnMajorR), false);
            }
          }
        }
      }
    } else if (warp == 1 && rank == 0) {
      // ---------------------------------------------------------- MMA issuer (leader CTA, converged warp)
      const bool lead = elect_one();
      begin();
      Ring<kStages> ring;
      auto wait_block = [&]() {
        if (!w.wait_warp(smem_u32(&sh->ready[ring.s]), ring.parity)) return false;
        tc_fence_after();
        return true;
      };
      // One elected lane issues a block's MMAs and the commit that frees the block in both CTAs.
      TileDesc rd{};                                 // of R and |R| of the tile in hand
      auto issue_rd = [&](uint32_t base, int kb, uint32_t idesc, uint32_t empty_bar) {
        const uint32_t ta = tmem_base + C::kColL + 64u * (kb & (kTmemStages - 1));
        if (lead) {
#pragma unroll
          for (int k = 0; k < kBlockK / 16; ++k)   // 16 bf16 = 32 bytes = 2 descriptor units = 8 columns of tensor memory per step
            mma_pair_a_tmem(tmem_base + C::kColRef, ta + 8u * k, rd.at(base + C::kOffR, k), idesc, k ? 1u : (uint32_t)kb, true);
#pragma unroll
          for (int k = 0; k < kBlockK / 16; ++k)
            mma_pair_a_tmem(tmem_base + C::kColDen, ta + 32u + 8u * k, rd.at(base + C::kOffRa, k), idesc, k ? 1u : (uint32_t)kb, true);
          tc_commit_pair(empty_bar, true);
        }
      };
      TileDesc cl{}, cr{};                           // of the codes of the variant in hand
      auto issue_lp = [&](auto kind, uint32_t base, uint32_t td, int kb, int steps, uint32_t idesc, uint32_t empty_bar) {
        if (lead) {
#pragma unroll
          for (int k = 0; k < C::kLpDepth / 32; ++k)
            if (k < steps)
              mma_pair<decltype(kind)::value>(td, cl.at(base + C::kOffL, k), cr.at(base + C::kOffR, k), idesc, k ? 1u : (uint32_t)kb, true);
          tc_commit_pair(empty_bar, true);
        }
      };
      uint32_t lp_uses0 = 0, lp_uses1 = 0;           // variants put into each 8-bit accumulator so far
      bool ok = true;
      uint32_t it = 0;
      for (int k = 0; k < sh->n_walk && ok; ++k) {
        const UnitInfo tw(sh->walk[k]);
        const bool r_mn = MN && (tw.major & kUnitMnMajorR);  // (A comes from tensor memory, contraction-major always)
        const uint32_t idesc_ref = make_idesc(1, 1, 1, kPairM, 2 * tw.half_n) | (r_mn ? kIdescMnMajorB : 0u);
        rd = tile_desc(r_mn, r_mn ? 2u * tw.half_n : 128u, 16u, 16u);
        const int nb = tw.lp_blocks();
        for (int j = 0; j < tw.n_tiles && ok; ++j, ++it) {
          // the reference and denominator blocks come back when both epilogues have copied the
          // previous tile's values out
          ok = it == 0 || w.wait_warp(smem_u32(&sh->rd_empty), (it - 1) & 1);
          if (!ok) break;
          tc_fence_after();
          for (int kb = 0; kb < tw.num_kb; ++kb) {
            ok = wait_block();
            if (!ok) break;
            issue_rd(tile_base + ring.s * C::kStageBytes, kb, idesc_ref, smem_u32(&sh->empty[ring.s]));
            ring.next();
          }
          if (!ok) break;
          tc_commit_pair(smem_u32(&sh->rd_full), lead);
          for (int f = 0; f < tw.n_var && ok; ++f) {
            const int b = (tw.n_var - 1 - f) & 1;
            const uint32_t idesc = __shfl_sync(0xffffffffu, sh->var[tw.var_begin + f].idesc, 0);
            const uint32_t flags = __shfl_sync(0xffffffffu, sh->var[tw.var_begin + f].flags, 0);
            const bool is_i8 = flags & kVarI8, cl_mn = MN && (flags & kVarMnMajorL), cr_mn = MN && (flags & kVarMnMajorR);
            cl = tile_desc(cl_mn, 128u, 32u, 16u);
            cr = tile_desc(cr_mn, cr_mn ? tw.half_n : 128u, 32u, 16u);
            // both epilogues have read what this accumulator held; the second one's columns have also
            // been this tile's L, which the denominator MMAs must have finished with
            const uint32_t uses = b ? lp_uses1 : lp_uses0;
            ok = uses == 0 || w.wait_warp(smem_u32(&sh->lp_done[b]), (uses - 1) & 1);
            if (ok && b == 1) ok = w.wait_warp(smem_u32(&sh->rd_full), it & 1);
            tc_fence_after();
            const uint32_t td = tmem_base + C::kColLp + 128u * b;
            for (int kb = 0; kb < nb && ok; ++kb) {
              ok = wait_block();
              if (!ok) break;
              const int steps = (tw.K - kb * C::kLpDepth + 31) / 32;          // of 32 codes; the rest of the block is fill
              const uint32_t base = tile_base + ring.s * C::kStageBytes, bar = smem_u32(&sh->empty[ring.s]);
              if (is_i8) issue_lp(std::integral_constant<int, kKindI8>{}, base, td, kb, steps, idesc, bar);
              else issue_lp(std::integral_constant<int, kKindF8>{}, base, td, kb, steps, idesc, bar);
              ring.next();
            }
            if (ok) tc_commit_pair(smem_u32(&sh->lp_full[b]), lead);
            if (b) ++lp_uses1; else ++lp_uses0;
          }
        }
      }
    } else if (RW && warp >= 2) {
      // ---------------------------------------------------------- |R| (both CTAs)
      begin();
      const int t = (warp - 2) * 32 + lane;        // 0..63
      const uint32_t ready_leader = map_to_cta(smem_u32(&sh->ready[0]), 0);
      Ring<kStages> ring;
      bool ok = true;
      for (int k = 0; k < sh->n_walk && ok; ++k)
        for (UnitInfo tw(sh->walk[k]); tw.n_tiles > 0 && ok; --tw.n_tiles) {
          for (int kb = 0; kb < tw.num_kb && ok; ++kb) {
            ok = w.wait_warp(smem_u32(&sh->full[ring.s]), ring.parity);
            if (!ok) break;
            abs_r<64>(tile_base + ring.s * C::kStageBytes + C::kOffR, C::kOffRa - C::kOffR, tw.half_n * 8, t);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(ready_leader + ring.s * 8u);
            ring.next();
          }
          const int n_code_blocks = tw.n_var * tw.lp_blocks();     // only passed on
          for (int kb = 0; kb < n_code_blocks && ok; ++kb) {
            ok = w.wait_warp(smem_u32(&sh->full[ring.s]), ring.parity);
            if (!ok) break;
            if (lane == 0) mbar_arrive_cluster(ready_leader + ring.s * 8u);
            ring.next();
          }
      }
    } else {
      begin();
    }
  } else if (warp < kFirstEpiWarp) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsConv));
    // ------------------------------------------------------------ converters (both CTAs)
    // Thread t of the four warps owns row t of this CTA's 128 left-operand rows (its warp's
    // tensor-memory lane quarter holds that row): once the stage has landed it reads its row of the
    // L tile from shared memory (128-byte swizzle: 16-byte chunk c of row r sits at c ^ (r & 7),
    // which makes these row-per-thread reads conflict-free) and stores the 32 words, and the same with
    // the sign bits cleared, into the stage's tensor-memory columns.  (Loading the rows with plain global loads
    // instead, to spare shared memory the 16 KB, was tried: a warp then touches 32 lines per
    // instruction and the converters became the bottleneck, 1.6 x slower overall.)
    const int q = warp & 3;
    const int t = q * 32 + lane;                   // 0..127
    const uint32_t ready_leader = map_to_cta(smem_u32(&sh->ready[0]), 0);
    const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + C::kColL;
    const uint32_t row_off = (uint32_t)t * 128u, sw = (uint32_t)t & 7u, m = 0x7fff7fffu;
    begin();
    Ring<kStages> ring;
    uint32_t it = 0, abs_uses = 0;                 // completions of abs_free awaited so far
    bool lent = false;                             // the previous tile's variants have used the L columns
    bool ok = true;
    for (int k = 0; k < sh->n_walk && ok; ++k)
      for (UnitInfo tw(sh->walk[k]); tw.n_tiles > 0 && ok; --tw.n_tiles, ++it) {
        // the L columns are free once the previous tile's denominator is complete and whatever
        // variants it put there have been read
        if (it > 0) ok = w.wait_warp(smem_u32(&sh->rd_full), (it - 1) & 1);
        if (ok && lent) ok = w.wait_warp(smem_u32(&sh->abs_free), abs_uses++ & 1);
        lent = tw.n_var > 1;
        const bool l_mn = MN && (tw.major & kUnitMnMajorL);
        // a loop for each order of L: one loop with the choice inside cost the contraction-major one 7 %
        auto convert = [&](auto mn) {
          constexpr bool kMn = decltype(mn)::value;
          for (int kb = 0; kb < tw.num_kb && ok; ++kb) {
            const uint32_t s = ring.s;
            ok = w.wait_warp(smem_u32(&sh->full[s]), ring.parity);
            if (!ok) break;
            const uint32_t base = tile_base + s * C::kStageBytes;
            if (!RW) abs_r<128>(base + C::kOffR, C::kOffRa - C::kOffR, tw.half_n * 8, t);
            uint32_t a[32];
            if constexpr (kMn) {
              load_l_mn_major(base + C::kOffL, q, lane, a);
            } else {
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const uint4 v = lds128(base + C::kOffL + row_off + (((uint32_t)j ^ sw) << 4));
                a[4 * j] = v.x; a[4 * j + 1] = v.y; a[4 * j + 2] = v.z; a[4 * j + 3] = v.w;
              }
            }
            if (kb >= kTmemStages) {
              // the tensor-memory columns were last read by the MMAs of the block kTmemStages before this one
              const uint32_t sp = s >= (uint32_t)kTmemStages ? s - kTmemStages : s + kStages - kTmemStages;
              const uint32_t pp = s >= (uint32_t)kTmemStages ? ring.parity : ring.parity ^ 1u;
              ok = w.wait_warp(smem_u32(&sh->empty[sp]), pp);
              if (!ok) break;
            }
            tc_fence_after();
            const uint32_t tcol = taddr + 64u * (uint32_t)(kb & (kTmemStages - 1));
            if constexpr (kMn) {
              tmem_st16x32(tcol, a);
              tmem_st16x32(tcol + (16u << 16), a + 16);
            } else {
              tmem_st32(tcol, a);
            }
#pragma unroll
            for (int j = 0; j < 32; ++j) a[j] &= m;
            if constexpr (kMn) {
              tmem_st16x32(tcol + 32u, a);
              tmem_st16x32(tcol + 32u + (16u << 16), a + 16);
            } else {
              tmem_st32(tcol + 32u, a);
            }
            if (!RW) fence_proxy_async();
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(ready_leader + s * 8u);
            ring.next();
          }
        };
        if (l_mn) convert(std::bool_constant<MN>{}); else convert(std::false_type{});
        // blocks of codes: only passed on
        const int n_code_blocks = tw.n_var * tw.lp_blocks();
        for (int kb = 0; kb < n_code_blocks && ok; ++kb) {
          ok = w.wait_warp(smem_u32(&sh->full[ring.s]), ring.parity);
          if (!ok) break;
          if (lane == 0) mbar_arrive_cluster(ready_leader + ring.s * 8u);
          ring.next();
        }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpi));
    // ------------------------------------------------------------ epilogue (warps 8..15, both CTAs)
    // A warp may touch the tensor-memory lane quarter warp % 4; the two warps of a quarter split
    // the columns.
    const int q = warp & 3;
    const int ew = warp - kFirstEpiWarp;           // 0..7
    const int h = ew >> 2;                         // which half of the tile's columns
    const int et = ew * 32 + lane;                 // 0..255
    const uint32_t rd_empty_leader = map_to_cta(smem_u32(&sh->rd_empty), 0);
    const uint32_t lp_done_leader = map_to_cta(smem_u32(&sh->lp_done[0]), 0);
    double acc_r2 = 0.0, acc_n2 = 0.0;             // of the unit in hand: sum C^2, D^2 of this thread's rows
    // reduce the statistics of the unit in hand over the CTA and write its records (all 256 threads call)
    auto flush = [&](int nv, int v0) {
      __syncwarp();                                // lanes 16..31 read below what lanes 0..15 have written to sums[]
      // values 3v, 3v + 1, 3v + 2: sum BE, max BE, sum diff^2 of variant v; the last two: sum C^2, D^2.  Half a warp adds up each
      for (int v = 0; v < nv; ++v) {
        const double2 a = sh->sums[v][ew][lane & 15];
        double x = lane < 16 ? a.x : a.y;
        const float mx = warp_max_f(sh->maxima[v][ew][lane & 15]);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) { sh->red[3 * v][ew] = x; sh->red[3 * v + 1][ew] = (double)mx; }
        if (lane == 16) sh->red[3 * v + 2][ew] = x;
      }
      const double rn = warp_sum4(acc_r2, acc_n2, 0.0, 0.0, lane);
      if (lane == 0) sh->red[3 * nv][ew] = rn;
      if (lane == 8) sh->red[3 * nv + 1][ew] = rn;
      acc_r2 = acc_n2 = 0.0;
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (et < 5 * nv) {
        const int v = et / 5, k = et - 5 * v;
        const int i = k < 3 ? 3 * v + k : 3 * nv + (k - 3);
        double x = 0.0;
        for (int j = 0; j < kEpiWarps; ++j) x = k == 1 ? fmax(x, sh->red[i][j]) : x + sh->red[i][j];
        __stcg(tab.v[v0 + v].partials + (int64_t)blockIdx.x * kPartialDoubles + k, x);
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");       // red[] may be reused
    };
    uint64_t met = 0;                              // bit v: this CTA has had tiles of probe v's unit
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
    uint32_t lp_parity = 0;                        // bit b: parity of the next use of 8-bit accumulator b
    // A wait for an 8-bit accumulator may run out in some warps and not in others (dead); the walk ends behind the barrier that
    // tells all of them (ended).  A warp that left by itself, at the end of a unit, would miss barriers that the others wait at.
    bool dead = false, ended = false;
    begin();
    uint32_t it = 0;
    for (int k = 0; k < sh->n_walk && !ended; ++k) {
      const UnitInfo tw(sh->walk[k]);
      const int pi = tw.unit, n_var = tw.n_var, v0 = tw.var_begin;
      met |= ((1ull << n_var) - 1ull) << v0;
      const int pM = tab.u[pi].M, pN = tab.u[pi].N;  // below 2^31 (its tensor maps require it)
      for (int v = 0; v < n_var; ++v)
        if (lane < 16) { sh->sums[v][ew][lane] = make_double2(0.0, 0.0); sh->maxima[v][ew][lane] = 0.f; }
      if (et < n_var) {                              // read after the barrier below
        const uint32_t flags = sh->var[v0 + et].flags;
        sh->dl_tensor[et] = flags & kVarScalePerRow ? 1.f : __ldg(tab.v[v0 + et].dl);
        sh->dr_tensor[et] = flags & kVarScalePerCol ? 1.f : __ldg(tab.v[v0 + et].dr);
      }
      for (int j = 0; j < tw.n_tiles; ++j, ++it) {
        const TileCoord tc = pair_tile(sh->walk[k], j, num_pairs);
        for (int v = 0; v < n_var; ++v) {
          if ((sh->var[v0 + v].flags & kVarScalePerCol) && et < kBlockN) {
            const int col = tc.n_tile * kBlockN + et;
            sh->delta_r[it & 1][v][et] = col < pN ? __ldg(tab.v[v0 + v].dr + (int64_t)tc.b * pN + col) : 0.f;
          }
        }
        const int row = tc.m_tile * kPairM + (int)rank * kBlockM + q * 32 + lane;
        const bool row_ok = row < pM;
        // the two warps of a lane quarter split the tile's columns: 64 each, or 32 each where the
        // tile is 64 wide (outputs at most 64 wide)
        const bool narrow = tw.half_n < 64;
        const int cw = narrow ? 32 : 64, cbase = h * cw;
        const int colw = tc.n_tile * kBlockN + cbase;                  // first column of this warp
        const int live = pN - colw < cw ? pN - colw : cw;              // its columns that exist; <= 0: none

        const bool ok = !dead && w.wait(smem_u32(&sh->rd_full), it & 1);
        // one barrier publishes the scales and makes the give-up decision uniform over the epilogue
        if (epi_barrier_any(!ok)) { ended = true; break; }
        tc_fence_after();
        uint32_t rc[64], rd[64];
        tmem_ld32(lane_addr + C::kColRef + cbase, *reinterpret_cast<uint32_t(*)[32]>(&rc[0]));
        tmem_ld32(lane_addr + C::kColDen + cbase, *reinterpret_cast<uint32_t(*)[32]>(&rd[0]));
        if (!narrow) {
          tmem_ld32(lane_addr + C::kColRef + cbase + 32, *reinterpret_cast<uint32_t(*)[32]>(&rc[32]));
          tmem_ld32(lane_addr + C::kColDen + cbase + 32, *reinterpret_cast<uint32_t(*)[32]>(&rd[32]));
        }
        tmem_ld_wait();
        // in registers: the MMA warp may start the next tile's reference and denominator as soon as
        // it is through with this tile's variants
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(rd_empty_leader);
        // sums of C^2 and D^2, and D replaced by its reciprocal (all under the first 8-bit product).
        // D == 0 implies C == Q == 0, so clamping the divisor keeps BE = 0 there without a branch.
        {
          uint64_t r22 = 0ull, n22 = 0ull;
          auto prepare = [&](int j0) {
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
              const uint64_t cv2 = pack2(__uint_as_float(rc[j0 + j]), __uint_as_float(rc[j0 + j + 1]));
              const float d0 = __uint_as_float(rd[j0 + j]), d1 = __uint_as_float(rd[j0 + j + 1]);
              const uint64_t dd2 = pack2(d0, d1);
              r22 = fma2(cv2, cv2, r22);
              n22 = fma2(dd2, dd2, n22);
              rd[j0 + j] = __float_as_uint(rcp_approx(fmaxf(d0, 1e-37f)));
              rd[j0 + j + 1] = __float_as_uint(rcp_approx(fmaxf(d1, 1e-37f)));
            }
          };
          if (live < cw) {                                 // ragged edge: columns beyond the matrix count as zeros
#pragma unroll
            for (int k = 0; k < 64; ++k)
              if (k >= live) { rc[k] = 0u; rd[k] = 0u; }
          }
          prepare(0);
          if (!narrow) prepare(32);
          float x0, x1;
          unpack2(r22, x0, x1);
          const double r2d = (double)x0 + (double)x1;
          unpack2(n22, x0, x1);
          const double n2d = (double)x0 + (double)x1;
          if (row_ok) {
            acc_r2 += r2d;
            acc_n2 += n2d;
            for (int v = 0; v < n_var; ++v) {
              if (!(sh->var[v0 + v].flags & kVarRowStats)) continue;       // the optional per-row check output
              double* const rs = tab.v[v0 + v].row_stats + ((int64_t)tc.b * pM + row) * 5;
              atomicAdd(rs + 3, r2d);
              atomicAdd(rs + 4, n2d);
            }
          }
        }
        for (int f = 0; f < n_var; ++f) {
          const int b = (n_var - 1 - f) & 1;
          const uint32_t flags = sh->var[v0 + f].flags;
          const bool per_col = (flags & kVarScalePerCol) != 0, is_i8 = (flags & kVarI8) != 0;
          float dlv = sh->dl_tensor[f];
          if (flags & kVarScalePerRow) dlv = row_ok ? __ldg(tab.v[v0 + f].dl + (int64_t)tc.b * pM + row) : 0.f;
          const float kd = per_col ? -dlv : -dlv * sh->dr_tensor[f];
          if (!w.wait_warp(smem_u32(&sh->lp_full[b]), (lp_parity >> b) & 1u)) { dead = true; break; }
          lp_parity ^= 1u << b;
          tc_fence_after();
          const uint32_t taddr = lane_addr + C::kColLp + 128u * b + cbase;
          StatsV st{0.f, 0.f, 0.f, 0ull};
          auto release = [&]() {
            // read to the end: the MMA warp may overwrite it and, after the tile's last use of the second
            // accumulator (once per tile, or the converters' wait could miss a phase of the barrier), this
            // CTA's converters may.  Every warp arrives exactly once per use.
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
              mbar_arrive_cluster(lp_done_leader + 8u * b);
              if (f == n_var - 2) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&sh->abs_free)) : "memory");
            }
          };
          if (per_col) eval_variant<true>(taddr, rc, rd, live, is_i8, pack2(kd, kd), sh->delta_r[it & 1][f] + cbase, st, release);
          else eval_variant<false>(taddr, rc, rd, live, is_i8, pack2(kd, kd), sh->delta_r[0][0], st, release);
          double be = 0.0, d2 = 0.0;
          float mx = 0.f;
          if (row_ok) {
            float x0, x1;
            unpack2(st.d2, x0, x1);
            be = (double)st.be0 + (double)st.be1;
            d2 = (double)x0 + (double)x1;
            mx = st.mx;
            if (flags & kVarRowStats) {
              double* const rs = tab.v[v0 + f].row_stats + ((int64_t)tc.b * pM + row) * 5;
              atomicAdd(rs + 0, be);
              atomicMax(reinterpret_cast<unsigned long long*>(rs + 1), (unsigned long long)__double_as_longlong((double)mx));
              atomicAdd(rs + 2, d2);
            }
          }
          be += __shfl_xor_sync(0xffffffffu, be, 16);
          d2 += __shfl_xor_sync(0xffffffffu, d2, 16);
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
          if (lane < 16) {
            double2& a = sh->sums[f][ew][lane];
            a.x += be;
            a.y += d2;
            sh->maxima[f][ew][lane] = fmaxf(sh->maxima[f][ew][lane], mx);
          }
        }
      }
      flush(n_var, v0);
    }
    // the records of the probes this CTA never met are zero
    for (int i = et; i < kPartialDoubles * tab.n_var; i += 256) {
      const int v = i / kPartialDoubles;
      if (!(met >> v & 1ull)) __stcg(tab.v[v].partials + (int64_t)blockIdx.x * kPartialDoubles + (i - v * kPartialDoubles), 0.0);
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    if (et == 0) {
      __threadfence();                            // after the barrier: covers the records that the other threads have written
      const uint32_t prev = atomicAdd(tab.done_counter, 1u);
      sh->is_last = prev == gridDim.x - 1 ? 1u : 0u;
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    if (sh->is_last) {
      __threadfence();
      write_results(tab, ew, lane);
    }
  }

  probe_exit<kStages>(sh, tab.wait_limit_ns, warp, rank, tmem_base);
}

// ------------------------------------------------------------------ the fused probe kernel, one probe per unit
// Units of one probe share nothing, so their three products run side by side, k-block by k-block: a stage
// holds the bf16 and the code tiles of 64 contraction entries and one commit frees it.  112 KB go through shared
// memory per k-block (36 by TMA, 44 of MMA operands, 32 by the converters) against the 96 of the
// products one after the other, but a tile has no phases: the converters run four blocks ahead
// across its end, the next tile's reference and denominator MMAs start while this one's last columns are evaluated, and
// the epilogue takes all three products in one sweep (the reciprocals beside the other arithmetic,
// the sums in registers) with one wait.  Short contractions are bound by that chain, and by fetching its instructions: what
// a tile runs once, all roles together, is more than the instruction cache holds beside the loops (512 x 512 x 64 x 256:
// stalls for instructions per issue 1.1 -> 2.7 with the code for mn-major operands and integer divisions in the walk, 98 ->
// 119 us; without either 102, with |R| written by the converters as well 94).  Measured, the fused kernel
// alone, one after the other / side by side: 512 x 512 x 64 x 256 131 / 88 us; 8192 x 4096 with K = 128 75 / 53,
// K = 256 76 / 64, K = 512 91 / 88, K = 1024 145 / 140.  With three probes per unit sharing wins from K = 64 on (187 / 239 us).
// |R| by the converters / by two warps of its own: 8192 x 4096 x 1024 160 / 141 us, 2048 x 3072 x 2048 76 / 69, 2048^2 x
// 16384 355 / 300 (short contractions the other way round: r_by_warps).  L from tensor memory as well (two stages of both, 96 KB) measured 140, 70 and 318, and 66 instead of
// 60 at K = 192, where two blocks are not enough ahead.
//   Roles, registers, walk and exit are those of tc_group_kernel.  Tensor memory: columns 0..127 reference, 128..255
// denominator, 256..383 the 8-bit product, 384..511 four stages of |L| (32 columns of two bf16 each).
struct CfgS {
  static constexpr int kStages = 5;          // stages of shared memory (TMA ring)
  static constexpr int kAbsStages = 4;       // stages of |L| in tensor memory (128 columns / 32)
  // stage: L, R, |R| (written by warps 2 and 3 or the converters), codes of L, codes of R
  static constexpr uint32_t kOffL = 0, kOffR = kABf16, kOffRa = kOffR + kBBf16, kOffCl = kOffRa + kBBf16;
  static constexpr uint32_t kOffCr = kOffCl + kALp;
  static constexpr uint32_t kStageBytes = kOffCr + kBLp;             // 44 KB
  static constexpr uint32_t kTileBytes = kStages * kStageBytes;      // 220 KB
  static constexpr uint32_t kColRef = 0, kColDen = 128, kColLp = 256, kColAbsL = 384;   // tensor-memory columns
};

template <int UNITS>
struct SharedS {
  uint64_t full[CfgS::kStages];     // per CTA: this CTA's loads of a stage have landed
  uint64_t ready[CfgS::kStages];    // leader: both CTAs' converters (and warps 2 and 3, with RW) have seen their loads
                                    //         land and have written |L| (tensor memory) and |R| (stage)
  uint64_t empty[CfgS::kStages];    // per CTA: the pair's MMAs have finished with the k-block of the stage
  uint64_t tmem_full;               // per CTA: the tile's accumulators are complete
  uint64_t tmem_empty;              // leader: both CTAs' epilogues have copied out reference and denominator
  uint64_t lp_done;                 // leader: both CTAs' epilogues have finished a tile
  uint64_t drain;                   // leader, give-up path only: every MMA issued so far has completed
  uint32_t tmem_base;
  uint32_t abort_flag;
  uint32_t is_last;
  uint32_t issued;                  // k-blocks whose loads the producer has issued (read on the give-up path)
  float delta_r[2][kBlockN];
  double red[4][kEpiWarps];
  float red_max[kEpiWarps];
  int32_t n_walk;                   // units that give this pair tiles
  WalkInfo walk[UNITS];
  VarInfo var[UNITS];               // of unit i: it has one probe
};

// Eq. 3 statistics of the side-by-side kernel, which first brings a chunk into one form (the 8-bit
// accumulator as fp32, dead columns zeroed) so that one instantiation per scale layout serves every
// format and the ragged edge.  PER_COL: the right operand has a scale per column
// (dr_s), otherwise kd2 holds (-delta_l delta_r) twice.
struct StatsG {
  float be0, be1;
  uint64_t d2, r2, n2;
  float mx;
};
template <bool PER_COL>
__device__ __forceinline__ void stats16g(const uint32_t* rc, const uint32_t* rd, const uint32_t* rq, uint64_t kd2,
                                         const float* dr_s, StatsG& s) {
#pragma unroll
  for (int j = 0; j < 16; j += 2) {
    const uint64_t a2 = pack2(__uint_as_float(rq[j]), __uint_as_float(rq[j + 1]));
    const uint64_t cv2 = pack2(__uint_as_float(rc[j]), __uint_as_float(rc[j + 1]));
    const float d0 = __uint_as_float(rd[j]), d1 = __uint_as_float(rd[j + 1]);
    const uint64_t dd2 = pack2(d0, d1);
    uint64_t diff2;                                              // C - A dl dr
    if (PER_COL) diff2 = fma2(mul2(a2, kd2), *reinterpret_cast<const uint64_t*>(dr_s + j), cv2);
    else diff2 = fma2(a2, kd2, cv2);
    // D == 0 implies C == Q == 0, so clamping the divisor keeps BE = 0 there without a branch
    const uint64_t be2 = mul2(diff2, pack2(rcp_approx(fmaxf(d0, 1e-37f)), rcp_approx(fmaxf(d1, 1e-37f))));
    float b0, b1;
    unpack2(be2, b0, b1);
    s.be0 += fabsf(b0);
    s.be1 += fabsf(b1);
    s.mx = fmaxf(s.mx, fmaxf(fabsf(b0), fabsf(b1)));
    s.d2 = fma2(diff2, diff2, s.d2);
    s.r2 = fma2(cv2, cv2, s.r2);
    s.n2 = fma2(dd2, dd2, s.n2);
  }
}
// Chunk CH (16 columns) of a warp's share of a tile: rq holds its 8-bit accumulators as read from
// tensor memory; n_live < 16 only at the ragged edge of the matrix, whose dead columns count as zeros.
template <int CH>
__device__ __forceinline__ void stats_chunk(uint32_t (&rc)[64], uint32_t (&rd)[64], uint32_t (&rq)[16], int n_live,
                                            bool is_i8, bool per_col, uint64_t kd2, const float* dr_s, StatsG& st) {
  if (is_i8) {
#pragma unroll
    for (int k = 0; k < 16; ++k) rq[k] = __float_as_uint((float)(int)rq[k]);
  }
  if (n_live < 16) {
#pragma unroll
    for (int k = 0; k < 16; ++k)
      if (k >= n_live) { rc[CH * 16 + k] = 0u; rd[CH * 16 + k] = 0u; rq[k] = 0u; }
  }
  if (per_col) stats16g<true>(&rc[CH * 16], &rd[CH * 16], rq, kd2, dr_s + CH * 16, st);
  else stats16g<false>(&rc[CH * 16], &rd[CH * 16], rq, kd2, nullptr, st);
}
// Adds one tile's share of a row's Eq. 3 sums to the optional per-row check output.
__device__ __forceinline__ void row_stats_add(double* rs, const StatsG& st) {
  float x0, x1;
  atomicAdd(rs + 0, (double)st.be0 + (double)st.be1);
  atomicMax(reinterpret_cast<unsigned long long*>(rs + 1), (unsigned long long)__double_as_longlong((double)st.mx));
  unpack2(st.d2, x0, x1); atomicAdd(rs + 2, (double)x0 + (double)x1);
  unpack2(st.r2, x0, x1); atomicAdd(rs + 3, (double)x0 + (double)x1);
  unpack2(st.n2, x0, x1); atomicAdd(rs + 4, (double)x0 + (double)x1);
}

// MN: units may have operands whose contraction is strided.  RW: |R| by warps of its own, not by the converters (r_by_warps).
template <typename Table, bool MN, bool RW>
__global__ void __launch_bounds__(kProbeThreads, 1)
tc_side_kernel(const __grid_constant__ Table tab) {
  using C = CfgS;
  using Sh = SharedS<Table::kUnits>;
  constexpr int kStages = C::kStages, kAbs = C::kAbsStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  Sh* sh = reinterpret_cast<Sh*>(tiles + C::kTileBytes);
  const uint32_t tile_base = smem_u32(tiles);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;
  const Waiter w{&sh->abort_flag, tab.err0, tab.wait_limit_ns};

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&sh->full[s]), 1);
      mbar_init(smem_u32(&sh->empty[s]), 1);
    }
    for (int s = 0; s < kStages; ++s) mbar_init(smem_u32(&sh->ready[s]), 2 * (RW ? 6 : 4));   // four converter warps and, with RW, two for |R| in each CTA
    mbar_init(smem_u32(&sh->tmem_full), 1);
    mbar_init(smem_u32(&sh->tmem_empty), 2 * kEpiWarps);
    mbar_init(smem_u32(&sh->lp_done), 2 * kEpiWarps);
    mbar_init(smem_u32(&sh->drain), 1);
    sh->abort_flag = 0;
    sh->is_last = 0;
    sh->issued = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&sh->tmem_base)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  if (warp == 2) fill_walk(sh, tab, lane, pair, num_pairs);
  tc_fence_before();
  __syncthreads();
  cluster_arrive();
  tc_fence_after();
  const uint32_t tmem_base = sh->tmem_base;
  auto begin = [&]() {
    cluster_wait();        // the peer's barriers and tensor memory exist before anyone uses them
    pdl_prologue();        // everything above overlapped the tail of the previous kernel
    tc_fence_after();
  };

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsCtl));
    if (warp == 0) {
      // ---------------------------------------------------------- TMA producer (both CTAs)
      begin();
      if (lane == 0) {
        Ring<kStages> ring;
        uint32_t g = 0;
        bool ok = true;
        for (int k = 0; k < sh->n_walk && ok; ++k) {
          const WalkInfo& wk = sh->walk[k];
          const int pi = wk.half_n >> 16;
          const CUtensorMap* const um = tab.unit_maps[pi];
          const CUtensorMap* const vm = tab.var_maps[pi];
          const int n_tiles = wk.n_tiles, num_kb = wk.num_kb, half_n = wk.half_n & 255;
          const uint32_t flags = sh->var[pi].flags, major = (uint32_t)wk.half_n >> 8 & 255u;
          const bool l_mn = MN && (major & kUnitMnMajorL), r_mn = MN && (major & kUnitMnMajorR);
          const bool cl_mn = MN && (flags & kVarMnMajorL), cr_mn = MN && (flags & kVarMnMajorR);
          for (int j = 0; j < n_tiles && ok; ++j) {
            const TileCoord tc = pair_tile(wk, j, num_pairs);
            const int r0 = tc.m_tile * kPairM + (int)rank * kBlockM;     // this CTA's left-operand rows
            const int c0 = tc.n_tile * kBlockN + (int)rank * half_n;     // this CTA's half of the right operand
            for (int kb = 0; kb < num_kb; ++kb, ++g) {
              const uint32_t s = ring.s;
              // test hook: the consumers' waits run out
              ok = g < tab.stop_after_kb && (g < (uint32_t)kStages || w.wait(smem_u32(&sh->empty[s]), ring.parity ^ 1u));
              if (!ok) break;
              const uint32_t bar = smem_u32(&sh->full[s]), base = tile_base + s * C::kStageBytes;
              mbar_expect_tx(bar, kABf16 + kALp + (uint32_t)half_n * (kBlockK * 2 + kBlockK));
              const int k0 = kb * kBlockK;
              tma_load_3d_local(base + C::kOffR, &um[1], bar, r_mn ? c0 : k0, r_mn ? k0 : c0, tc.b);
              tma_load_3d_local(base + C::kOffL, &um[0], bar, l_mn ? r0 : k0, l_mn ? k0 : r0, tc.b);
              if (l_mn) tma_load_3d_local(base + C::kOffL + kABf16 / 2, &um[0], bar, r0 + 64, k0, tc.b);
              tma_load_3d_local(base + C::kOffCl, &vm[0], bar, cl_mn ? r0 : k0, cl_mn ? k0 : r0, tc.b);
              tma_load_3d_local(base + C::kOffCr, &vm[1], bar, cr_mn ? c0 : k0, cr_mn ? k0 : c0, tc.b);
              sh->issued = g + 1;
              ring.next();
            }
          }
        }
      }
    } else if (warp == 1 && rank == 0) {
      // ---------------------------------------------------------- MMA issuer (leader CTA, converged warp)
      const bool lead = elect_one();
      uint32_t idesc_ref = 0, idesc_den = 0;   // of the tile in hand
      TileDesc ld{}, rd{}, cl{}, cr{};         // L; R and |R|; codes
      auto issue_ref_den = [&](uint32_t s, uint32_t gg, int kb) {
        const uint32_t base = tile_base + s * C::kStageBytes;
#pragma unroll
        for (int k = 0; k < kBlockK / 16; ++k)   // 16 bf16 per step
          mma_pair<kKindF16>(tmem_base + C::kColRef, ld.at(base + C::kOffL, k), rd.at(base + C::kOffR, k), idesc_ref, (kb | k) != 0, lead);
        const uint32_t ta = tmem_base + C::kColAbsL + 32u * (gg % kAbs);
#pragma unroll
        for (int k = 0; k < kBlockK / 16; ++k)   // 16 bf16 = 8 columns of tensor memory per step
          mma_pair_a_tmem(tmem_base + C::kColDen, ta + 8u * k, rd.at(base + C::kOffRa, k), idesc_den, (kb | k) != 0, lead);
      };
      auto issue_lp = [&](uint32_t s, int kb, bool is_i8, uint32_t idesc_lp) {
        const uint32_t base = tile_base + s * C::kStageBytes;
#pragma unroll
        for (int k = 0; k < kBlockK / 32; ++k) {  // 32 codes per step
          const uint64_t a = cl.at(base + C::kOffCl, k), b = cr.at(base + C::kOffCr, k);
          if (is_i8) mma_pair<kKindI8>(tmem_base + C::kColLp, a, b, idesc_lp, (kb | k) != 0, lead);
          else mma_pair<kKindF8>(tmem_base + C::kColLp, a, b, idesc_lp, (kb | k) != 0, lead);
        }
      };
      auto wait_stage = [&](const Ring<kStages>& at) {
        if (!w.wait_warp(smem_u32(&sh->ready[at.s]), at.parity)) return false;
        tc_fence_after();
        return true;
      };
      begin();
      Ring<kStages> ring;                      // of the next block whose 8-bit MMAs are to be issued
      uint32_t g = 0, it = 0;
      bool ok = true;
      for (int k = 0; k < sh->n_walk && ok; ++k) {
        const UnitInfo tw(sh->walk[k]);
        const int pi = tw.unit;
        const int num_kb = tw.num_kb;
        const uint32_t idesc_lp = __shfl_sync(0xffffffffu, sh->var[pi].idesc, 0);
        const uint32_t flags = __shfl_sync(0xffffffffu, sh->var[pi].flags, 0);
        const bool is_i8 = flags & kVarI8;
        const bool l_mn = MN && (tw.major & kUnitMnMajorL), r_mn = MN && (tw.major & kUnitMnMajorR);
        const bool cl_mn = MN && (flags & kVarMnMajorL), cr_mn = MN && (flags & kVarMnMajorR);
        // |L| comes from tensor memory, contraction-major always
        idesc_den = make_idesc(1, 1, 1, kPairM, 2 * tw.half_n) | (r_mn ? kIdescMnMajorB : 0u);
        idesc_ref = idesc_den | (l_mn ? kIdescMnMajorA : 0u);
        ld = tile_desc(l_mn, 128u, 16u, kABf16 / 2);
        rd = tile_desc(r_mn, r_mn ? 2u * tw.half_n : 128u, 16u, 16u);
        cl = tile_desc(cl_mn, cl_mn ? 128u : 64u, 32u, 16u);
        cr = tile_desc(cr_mn, cr_mn ? tw.half_n : 64u, 32u, 16u);
        for (int j = 0; j < tw.n_tiles && ok; ++j, ++it) {
          // the reference and denominator blocks come back when both epilogues have copied the
          // previous tile's values out; the 8-bit block when they have finished that tile
          ok = it == 0 || w.wait_warp(smem_u32(&sh->tmem_empty), (it - 1) & 1);
          if (!ok) break;
          tc_fence_after();
          const int n_ahead = num_kb < kAbs ? num_kb : kAbs;
          Ring<kStages> ahead = ring;
          for (int i = 0; i < n_ahead && ok; ++i) {
            ok = wait_stage(ahead);
            if (ok) issue_ref_den(ahead.s, g + i, i);
            ahead.next();
          }
          if (!ok) break;
          ok = it == 0 || w.wait_warp(smem_u32(&sh->lp_done), (it - 1) & 1);
          if (!ok) break;
          tc_fence_after();
          int kb = 0;
          for (; kb < n_ahead; ++kb, ++g) {
            issue_lp(ring.s, kb, is_i8, idesc_lp);
            tc_commit_pair(smem_u32(&sh->empty[ring.s]), lead);
            ring.next();
          }
          for (; kb < num_kb && ok; ++kb, ++g) {
            ok = wait_stage(ring);
            if (!ok) break;
            issue_ref_den(ring.s, g, kb);
            issue_lp(ring.s, kb, is_i8, idesc_lp);
            tc_commit_pair(smem_u32(&sh->empty[ring.s]), lead);             // frees the k-block in both CTAs
            ring.next();
          }
          if (ok) tc_commit_pair(smem_u32(&sh->tmem_full), lead);           // this tile's accumulators are complete
        }
      }
    } else if (RW && warp >= 2) {
      // ---------------------------------------------------------- |R| (both CTAs)
      begin();
      const int t = (warp - 2) * 32 + lane;        // 0..63
      const uint32_t ready_leader = map_to_cta(smem_u32(&sh->ready[0]), 0);
      bool ok = true;
      Ring<kStages> ring;
      for (int k = 0; k < sh->n_walk && ok; ++k)
        for (UnitInfo tw(sh->walk[k]); tw.n_tiles > 0 && ok; --tw.n_tiles) {
          for (int kb = 0; kb < tw.num_kb; ++kb) {
            ok = w.wait_warp(smem_u32(&sh->full[ring.s]), ring.parity);
            if (!ok) break;
            abs_r<64>(tile_base + ring.s * C::kStageBytes + C::kOffR, C::kOffRa - C::kOffR, tw.half_n * 8, t);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(ready_leader + ring.s * 8u);
            ring.next();
          }
      }
    } else {
      begin();
    }
  } else if (warp < kFirstEpiWarp) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsConv));
    // ------------------------------------------------------------ converters (both CTAs)
    // As in tc_group_kernel, but only |L| goes to tensor memory (the reference MMAs read L from shared memory),
    // and the k-blocks are counted through over all tiles: the converters run up to kAbs blocks ahead
    // of the MMAs across a tile's end.
    const int q = warp & 3;
    const int t = q * 32 + lane;                   // 0..127
    const uint32_t ready_leader = map_to_cta(smem_u32(&sh->ready[0]), 0);
    const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + C::kColAbsL;
    const uint32_t row_off = (uint32_t)t * 128u, sw = (uint32_t)t & 7u;
    begin();
    bool ok = true;
    Ring<kStages> ring;
    uint32_t g = 0;
    // the blocks of one tile; a loop for each order of L: one loop with the choice inside cost the contraction-major one 7 %
    auto convert = [&](auto mn, const UnitInfo& tw) {
      constexpr bool kMn = decltype(mn)::value;
      for (int kb = 0; kb < tw.num_kb; ++kb, ++g) {
        const uint32_t s = ring.s, m = 0x7fff7fffu;
        if (!w.wait_warp(smem_u32(&sh->full[s]), ring.parity)) { ok = false; return; }
        const uint32_t base = tile_base + s * C::kStageBytes;
        if (!RW) abs_r<128>(base + C::kOffR, C::kOffRa - C::kOffR, tw.half_n * 8, t);
        uint32_t a[32];
        if constexpr (kMn) {
          load_l_mn_major(base + C::kOffL, q, lane, a);
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint4 v = lds128(base + C::kOffL + row_off + (((uint32_t)j ^ sw) << 4));
            a[4 * j] = v.x; a[4 * j + 1] = v.y; a[4 * j + 2] = v.z; a[4 * j + 3] = v.w;
          }
        }
        // the tensor-memory columns were last read by the MMAs of k-block g - kAbs
        if (g >= (uint32_t)kAbs) {
          const uint32_t sp = s >= (uint32_t)kAbs ? s - kAbs : s + kStages - kAbs;
          const uint32_t pp = s >= (uint32_t)kAbs ? ring.parity : ring.parity ^ 1u;
          if (!w.wait_warp(smem_u32(&sh->empty[sp]), pp)) { ok = false; return; }
        }
        tc_fence_after();
        const uint32_t tcol = taddr + 32u * (g % kAbs);
#pragma unroll
        for (int j = 0; j < 32; ++j) a[j] &= m;
        if constexpr (kMn) {
          tmem_st16x32(tcol, a);
          tmem_st16x32(tcol + (16u << 16), a + 16);
        } else {
          tmem_st32(tcol, a);
        }
        if (!RW) fence_proxy_async();
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(ready_leader + s * 8u);
        ring.next();
      }
    };
    for (int k = 0; k < sh->n_walk && ok; ++k)
      for (UnitInfo tw(sh->walk[k]); tw.n_tiles > 0 && ok; --tw.n_tiles) {
        if (MN && (tw.major & kUnitMnMajorL)) convert(std::bool_constant<MN>{}, tw); else convert(std::false_type{}, tw);
      }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpi));
    // ------------------------------------------------------------ epilogue (warps 8..15, both CTAs)
    // A warp may touch the tensor-memory lane quarter warp % 4; the two warps of a quarter split
    // the columns.  Copy this warp's 64 columns of the reference and denominator blocks into
    // registers, hand those two blocks back to the MMA lane, then walk the 8-bit block in chunks
    // of 16 columns; the statistics arithmetic runs under the next tile's main loop.
    const int q = warp & 3;
    const int ew = warp - kFirstEpiWarp;           // 0..7
    const int h = ew >> 2;                         // which half of the tile's columns
    const int et = ew * 32 + lane;                 // 0..255
    const uint32_t tmem_empty_leader = map_to_cta(smem_u32(&sh->tmem_empty), 0);
    double acc[4] = {0, 0, 0, 0};                  // of the unit in hand: sum BE, sum diff^2, C^2, D^2
    float acc_max = 0.f;                           // and max BE
    // reduce the statistics of unit `pi` over the CTA and write its record (all 256 threads call)
    auto flush = [&](int pi) {
      const double x = warp_sum4(acc[0], acc[1], acc[2], acc[3], lane);
      const float mx = warp_max_f(acc_max);
      if ((lane & 7) == 0) sh->red[lane >> 3][ew] = x;
      if (lane == 0) sh->red_max[ew] = mx;
      acc[0] = acc[1] = acc[2] = acc[3] = 0.0;
      acc_max = 0.f;
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (ew == 0) {                               // lanes 8 k .. 8 k + 7: the warps' sums of value k
        double y = sh->red[lane >> 3][lane & 7];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
        const float m = warp_max_f(sh->red_max[lane & 7]);
        double* const rec = tab.v[pi].partials + (int64_t)blockIdx.x * kPartialDoubles;
        if ((lane & 7) == 0) __stcg(rec + (lane == 0 ? 0 : (lane >> 3) + 1), y);
        if (lane == 1) __stcg(rec + 1, (double)m);
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");       // red[] may be reused
    };
    uint32_t met = 0;                              // bit pi: this CTA has had tiles of unit pi
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
    // Of the unit in hand, read with its first tile.  Read ahead of the loop over tiles, as tc_group_kernel does, they are known not to change in it, and
    // the loop is compiled for each of their cases: 512 x 512 x 64 x 256 70.6 us so, 82.5 then, 78 with the tiles dealt in rounds.
    int cur = -1;                                  // the unit in hand
    bool per_col = false, pc_l = false, is_i8 = false, narrow = false;
    float dr_tensor = 1.f, dl_tensor = 0.f;
    int pM = 0, pN = 0;                            // below 2^31 (its tensor maps require it)
    begin();
    uint32_t it = 0;
    bool dead = false;                             // a wait ran out
    for (int k = 0; k < sh->n_walk && !dead; ++k) {
      const UnitInfo tw(sh->walk[k]);
      const int pi = tw.unit;
      for (int j = 0; j < tw.n_tiles; ++j, ++it) {
        if (pi != cur) {
          if (cur >= 0) flush(cur);
          cur = pi;
          met |= 1u << pi;
          const uint32_t flags = sh->var[pi].flags;
          per_col = flags & kVarScalePerCol; pc_l = flags & kVarScalePerRow; is_i8 = flags & kVarI8; narrow = tw.half_n < 64;
          pM = tab.u[pi].M; pN = tab.u[pi].N;
          dr_tensor = per_col ? 1.f : __ldg(tab.v[pi].dr);
          dl_tensor = pc_l ? 0.f : __ldg(tab.v[pi].dl);
        }
        const TileCoord tc = pair_tile(sh->walk[k], j, num_pairs);
        float* dr_s = sh->delta_r[it & 1];
        if (per_col && et < kBlockN) {
          const int col = tc.n_tile * kBlockN + et;
          dr_s[et] = col < pN ? __ldg(tab.v[pi].dr + (int64_t)tc.b * pN + col) : 0.f;
        }
        const int row = tc.m_tile * kPairM + (int)rank * kBlockM + q * 32 + lane;
        const bool row_ok = row < pM;
        float dlv = dl_tensor;
        if (pc_l) dlv = row_ok ? __ldg(tab.v[pi].dl + (int64_t)tc.b * pM + row) : 0.f;
        // the two warps of a lane quarter split the tile's columns: 64 each, or 32 each where the
        // tile is 64 wide (outputs at most 64 wide)
        const int cw = narrow ? 32 : 64, cbase = h * cw;
        const int colw = tc.n_tile * kBlockN + cbase;                  // first column of this warp

        const bool ok = w.wait(smem_u32(&sh->tmem_full), it & 1);
        // one barrier publishes delta_r and makes the give-up decision uniform over the epilogue
        if (epi_barrier_any(!ok)) { dead = true; break; }
        tc_fence_after();
        // live = columns of this warp that exist in the matrix
        const int live = pN - colw < cw ? pN - colw : cw;          // <= 0: none
        const uint32_t lp_addr = lane_addr + C::kColLp + cbase;
        const uint32_t lp_done_leader = map_to_cta(smem_u32(&sh->lp_done), 0);
        const float* const drc = dr_s + cbase;
        uint32_t rc[64], rd[64], rq0[16];
        tmem_ld32(lane_addr + C::kColRef + cbase, *reinterpret_cast<uint32_t(*)[32]>(&rc[0]));
        tmem_ld32(lane_addr + C::kColDen + cbase, *reinterpret_cast<uint32_t(*)[32]>(&rd[0]));
        if (!narrow) {
          tmem_ld32(lane_addr + C::kColRef + cbase + 32, *reinterpret_cast<uint32_t(*)[32]>(&rc[32]));
          tmem_ld32(lane_addr + C::kColDen + cbase + 32, *reinterpret_cast<uint32_t(*)[32]>(&rd[32]));
        }
        if (live > 0) tmem_ld16(lp_addr, rq0);
        tmem_ld_wait();
        // The reference and denominator blocks are in registers: the MMA lane may start the next
        // tile's bf16 MMAs.  The 8-bit block follows in two steps, its first 16 columns with the
        // loads above and the rest once the first chunk has been evaluated (which frees the
        // registers the rest is read into); then the MMA lane may start the next tile's 8-bit MMAs as well, while the
        // remaining chunks are still being evaluated.  Every warp arrives on each barrier exactly
        // once per tile.
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive_cluster(tmem_empty_leader);
          if (live <= 16) mbar_arrive_cluster(lp_done_leader);      // nothing further to read
        }
        StatsG st{0.f, 0.f, 0ull, 0ull, 0ull, 0.f};
        const float kd = -dlv * dr_tensor;
        const uint64_t kd2 = per_col ? pack2(-dlv, -dlv) : pack2(kd, kd);
        if (live > 0) stats_chunk<0>(rc, rd, rq0, live, is_i8, per_col, kd2, drc, st);
        if (live > 16) {
          // chunk 1 into the first chunk's registers, chunks 2 and 3 into those of the first
          // chunk's reference and denominator values
          uint32_t(&rq2)[16] = *reinterpret_cast<uint32_t(*)[16]>(&rc[0]);
          uint32_t(&rq3)[16] = *reinterpret_cast<uint32_t(*)[16]>(&rd[0]);
          tmem_ld16(lp_addr + 16, rq0);
          if (live > 32) tmem_ld16(lp_addr + 32, rq2);
          if (live > 48) tmem_ld16(lp_addr + 48, rq3);
          tmem_ld_wait();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(lp_done_leader);
          stats_chunk<1>(rc, rd, rq0, live - 16, is_i8, per_col, kd2, drc, st);
          if (live > 32) stats_chunk<2>(rc, rd, rq2, live - 32, is_i8, per_col, kd2, drc, st);
          if (live > 48) stats_chunk<3>(rc, rd, rq3, live - 48, is_i8, per_col, kd2, drc, st);
        }
        if (row_ok) {
          float x0, x1;
          acc[0] += (double)st.be0 + (double)st.be1;
          unpack2(st.d2, x0, x1); acc[1] += (double)x0 + (double)x1;
          unpack2(st.r2, x0, x1); acc[2] += (double)x0 + (double)x1;
          unpack2(st.n2, x0, x1); acc[3] += (double)x0 + (double)x1;
          acc_max = fmaxf(acc_max, st.mx);
          double* const rows = tab.v[pi].row_stats;
          if (rows) row_stats_add(rows + ((int64_t)tc.b * pM + row) * 5, st);
        }
      }
    }
    if (cur >= 0) flush(cur);
    // the records of the probes this CTA never met are zero
    if (et == 0) {
      for (int pi = 0; pi < tab.n; ++pi) {
        if (met & (1u << pi)) continue;
        double* rec = tab.v[pi].partials + (int64_t)blockIdx.x * kPartialDoubles;
        for (int i = 0; i < 5; ++i) __stcg(rec + i, 0.0);
      }
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    if (et == 0) {
      __threadfence();
      const uint32_t prev = atomicAdd(tab.done_counter, 1u);
      sh->is_last = prev == gridDim.x - 1 ? 1u : 0u;
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    if (sh->is_last) {
      __threadfence();
      write_results(tab, ew, lane);
    }
  }

  probe_exit<kStages>(sh, tab.wait_limit_ns, warp, rank, tmem_base);
}

// ------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// Tensor map over [batch][rows][K] with the contracting index contiguous; box = 64 x box_rows x 1,
// swizzle span = row width of the box (128 bytes for bf16, 64 bytes for codes).
// wide: 128-byte boxes and swizzle for the codes as well (the 256 x 256 tile kernel).
bool make_map(CUtensorMap* m, const void* base, bool bf16, int box_rows, int64_t K, int64_t rows, int64_t batch,
              int64_t ld_elems, int64_t sb_elems, bool wide = false) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const uint64_t es = bf16 ? 2 : 1;
  cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)batch};
  cuuint64_t sb = batch > 1 ? (cuuint64_t)sb_elems * es : (cuuint64_t)rows * ld_elems * es;
  cuuint64_t strides[2] = {(cuuint64_t)ld_elems * es, sb};
  cuuint32_t box[3] = {(cuuint32_t)((wide && !bf16) ? 2 * kBlockK : kBlockK), (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(m, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 3,
                  const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  (bf16 || wide) ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// The same over [batch][K][rows] with the operand's rows contiguous (contraction strided): box = box_rows x depth x 1, whose
// rows of box_rows elements are one swizzle span (32, 64 or 128 bytes).
bool make_map_mn(CUtensorMap* m, const void* base, bool bf16, int box_rows, int depth, int64_t K, int64_t rows, int64_t batch,
                   int64_t ld_elems, int64_t sb_elems) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const uint64_t es = bf16 ? 2 : 1;
  cuuint64_t dims[3] = {(cuuint64_t)rows, (cuuint64_t)K, (cuuint64_t)batch};
  cuuint64_t strides[2] = {(cuuint64_t)ld_elems * es, batch > 1 ? (cuuint64_t)sb_elems * es : (cuuint64_t)K * ld_elems * es};
  cuuint32_t box[3] = {(cuuint32_t)box_rows, (cuuint32_t)depth, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  const uint64_t span = box_rows * es;
  CUresult r = fn(m, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 3,
                  const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  span == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : span == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

uint32_t lp_idesc(int fmt_l, int fmt_r, int n = kBlockN) {
  if (fmt_l == QM_FMT_INT8) return make_idesc(2, 1, 1, kPairM, n);                 // s8 x s8 -> s32
  const uint32_t fa = fmt_l == QM_FMT_E4M3 ? 0u : 1u, fb = fmt_r == QM_FMT_E4M3 ? 0u : 1u;
  return make_idesc(1, fa, fb, kPairM, n);                                         // fp8 x fp8 -> f32
}

template <int MODE>
size_t smem_bytes() {
  // the plain products' output goes out through 4 KB per epilogue warp, behind the control block
  return (size_t)Cfg<MODE>::kStages * Cfg<MODE>::kStageBytes + sizeof(Shared) + 1024 + (MODE == kProbe2 ? 0 : kEpiWarps * 4096);
}

int64_t tile_count(GemmShape g) {
  return ((g.M + kPairM - 1) / kPairM) * ((g.N + kBlockN - 1) / kBlockN) * g.batch;
}

bool shape_ok(GemmShape g) {
  if (!(g.M > 0 && g.N > 0 && g.K > 0 && g.batch > 0 && (g.K % 16) == 0)) return false;
  // row, column and contraction indices of a tile's far edge are formed in 32-bit integers
  constexpr int64_t kLimit = (1ll << 31) - 1024;
  if (g.M >= kLimit || g.N >= kLimit || g.K >= kLimit || g.batch >= (1ll << 31)) return false;
  return tile_count(g) < (1ll << 31);
}

void fill_tiles(KernelArgs* ka, GemmShape g) {
  ka->M = g.M; ka->N = g.N; ka->K = g.K;
  ka->tiles_m = (int32_t)((g.M + kPairM - 1) / kPairM);
  ka->tiles_n = (int32_t)((g.N + kBlockN - 1) / kBlockN);
  ka->num_tiles = (int32_t)tile_count(g);
}

// CTA pairs that can be resident at once (one per TPC unless the device says fewer).
int g_max_pairs[kMaxDevices] = {};     // per device; 0 = not yet queried
int max_pairs() {
  const int dev = current_device();
  return dev >= 0 && g_max_pairs[dev] > 0 ? g_max_pairs[dev] : std::min(sm_count() / 2, kMaxPairs);
}

// cudaFuncSetAttribute(MaxDynamicSharedMemorySize) once per kernel and device.
template <typename K>
qm_status allow_smem(K kern, size_t bytes, bool (&done)[kMaxDevices]) {
  const int dev = current_device();
  if (dev < 0) return QM_ERR_UNSUPPORTED;
  if (!done[dev]) {
    QM_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    done[dev] = true;
  }
  return QM_OK;
}

// CTAs to launch: two per tile, at most the resident number of pairs.
int grid_size(GemmShape g) {
  const int64_t tiles = tile_count(g);
  const int pairs = max_pairs();
  return 2 * (int)(tiles < pairs ? tiles : pairs);
}

// maps: eight tensor maps (L, R, |L|, |R|, codes L, codes R, second-format codes L, R).
template <int MODE, int LPKIND, int LPKIND2 = LPKIND>
qm_status launch(const CUtensorMap* maps, const KernelArgs& ka, GemmShape g, cudaStream_t s) {
  auto kern = tc_kernel<MODE, LPKIND, LPKIND2>;
  static bool attr_done[kMaxDevices] = {};     // per instantiation
  const qm_status as = allow_smem(kern, smem_bytes<MODE>(), attr_done);
  if (as != QM_OK) return as;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid_size(g));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem_bytes<MODE>();
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // see pdl_prologue()
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 2 : 1;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  if (MODE == kProbe2) profile_events(&ev0, &ev1);
  if (ev0) QM_CUDA_OK(cudaEventRecord(ev0, s));
  QM_CUDA_OK(cudaLaunchKernelEx(&cfg, kern, maps[0], maps[1], maps[2], maps[3], maps[4], maps[5], maps[6], maps[7],
                                ka));
  if (ev1) QM_CUDA_OK(cudaEventRecord(ev1, s));
  count_launch();
  return QM_OK;
}

// The 256 x 256 tile kernel: worth it once the output is at least one such tile wide.
bool use_wide(GemmShape g) { return g.N >= kWideN; }

template <int KIND>
qm_status launch_wide(const CUtensorMap& ma, const CUtensorMap& mb, KernelArgs ka, GemmShape g, cudaStream_t s) {
  auto kern = tc_gemm_wide_kernel<KIND>;
  constexpr size_t smem = (size_t)kWideStages * kWideStageBytes + sizeof(SharedWide) + 1024;
  static bool attr_done[kMaxDevices] = {};
  const qm_status as = allow_smem(kern, smem, attr_done);
  if (as != QM_OK) return as;
  ka.tiles_m = (int32_t)((g.M + kPairM - 1) / kPairM);
  ka.tiles_n = (int32_t)((g.N + kWideN - 1) / kWideN);
  const int64_t tiles = (int64_t)ka.tiles_m * ka.tiles_n * g.batch;
  if (tiles >= (1ll << 31)) return QM_ERR_UNSUPPORTED;
  ka.num_tiles = (int32_t)tiles;
  const int pairs = max_pairs();
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(2 * (tiles < pairs ? tiles : pairs)));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 2 : 1;
  QM_CUDA_OK(cudaLaunchKernelEx(&cfg, kern, ma, mb, ka));
  count_launch();
  return QM_OK;
}

}  // namespace

namespace {
// The two forms of the fused kernel, units of one probe (SIDE) and units of several, each with and without operands whose
// contraction is strided: what those need is a third of the roles' code, and short tiles wait for instructions (below).
template <bool SIDE, bool MN, bool RW, typename Table>
struct ProbeKernel {
  static constexpr auto kernel = SIDE ? tc_side_kernel<Table, MN, RW> : tc_group_kernel<Table, MN, RW>;
  static constexpr size_t kSmem = 1024 + (SIDE ? (size_t)CfgS::kTileBytes + sizeof(SharedS<Table::kUnits>)
                                               : (size_t)CfgP::kTileBytes + sizeof(SharedP<Table::kUnits, Table::kVars>));
  static_assert(kSmem <= 232448, "shared memory of a CTA");
};

// Bound of the fused kernels' barrier waits and the producer's test hook (see qm_debug_* in qm.h).
std::atomic<uint64_t> g_wait_limit_ns{1000000000ull};
std::atomic<uint32_t> g_stop_after_kb{0xffffffffu};

template <typename PK>
qm_status probe_kernel_ready() {
  static bool attr_done[kMaxDevices] = {};
  const int dev = current_device();
  if (dev < 0) return QM_ERR_UNSUPPORTED;
  if (!attr_done[dev]) {
    // the kernel re-divides the registers its block was launched with (setmaxnreg): refuse to
    // launch if the compiler gave it fewer than the split adds up to, because an increase that
    // cannot be served waits forever
    cudaFuncAttributes fa{};
    QM_CUDA_OK(cudaFuncGetAttributes(&fa, PK::kernel));
    if (fa.numRegs * 4 < kRegsCtl + kRegsConv + 2 * kRegsEpi) return QM_ERR_UNSUPPORTED;
  }
  return allow_smem(PK::kernel, PK::kSmem, attr_done);
}

template <bool SIDE, typename Table>
qm_status probe_kernels_ready() {
  qm_status st = probe_kernel_ready<ProbeKernel<SIDE, false, false, Table>>();
  if (st == QM_OK) st = probe_kernel_ready<ProbeKernel<SIDE, false, true, Table>>();
  if (st == QM_OK) st = probe_kernel_ready<ProbeKernel<SIDE, true, false, Table>>();
  if (st == QM_OK) st = probe_kernel_ready<ProbeKernel<SIDE, true, true, Table>>();
  return st;
}

// CTA pairs of the fused probe kernel that can be resident at once (its footprint is the largest
// of all modes, so its residency bounds every grid); queried once per device.
qm_status probe_residency() {
  const int dev = current_device();
  if (dev < 0) return QM_ERR_UNSUPPORTED;
  using Widest = ProbeKernel<false, true, true, TableBig>;
  qm_status as = probe_kernels_ready<false, TableBig>();
  if (as == QM_OK) as = probe_kernels_ready<true, TableBig>();
  if (as == QM_OK) as = probe_kernels_ready<true, TableOne>();
  if (as != QM_OK) return as;
  if (g_max_pairs[dev] == 0) {
    cudaLaunchConfig_t q{};
    q.gridDim = dim3((unsigned)(2 * (sm_count() / 2))); q.blockDim = dim3(kProbeThreads);
    q.dynamicSmemBytes = Widest::kSmem;
    cudaLaunchAttribute qa[1];
    qa[0].id = cudaLaunchAttributeClusterDimension;
    qa[0].val.clusterDim.x = 2; qa[0].val.clusterDim.y = 1; qa[0].val.clusterDim.z = 1;
    q.attrs = qa; q.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, Widest::kernel, &q) == cudaSuccess && n > 0)
      g_max_pairs[dev] = std::min(n, std::min(sm_count() / 2, kMaxPairs));
    else
      g_max_pairs[dev] = std::min(sm_count() / 2, kMaxPairs);
    (void)cudaGetLastError();
  }
  return QM_OK;
}

// The probes of one unit, by their index in the caller's list.
struct UnitPlan {
  GemmShape g;
  int n_var;
  int probe[kMaxVar];
  double cycles;              // of a tile (tile_cycles)
};

bool same_products(const TcProbeArgs& a, const TcProbeArgs& b) {
  return a.l == b.l && a.l_ld == b.l_ld && a.l_sb == b.l_sb && a.r == b.r && a.r_ld == b.r_ld && a.r_sb == b.r_sb &&
         a.l_mn == b.l_mn && a.r_mn == b.r_mn && a.g.M == b.g.M && a.g.N == b.g.N && a.g.K == b.g.K && a.g.batch == b.g.batch;
}

// Whether |R| gets two warps of its own.  Long contractions wait for the converters, short ones for the epilogue and for
// instructions, which the role adds to: with one probe to a unit up to two blocks of the contraction, with several up to as
// many as the ring has stages.  Whole batches in us, |R| by the converters / by warps of its own: one format 512 x 512 x 64 x 256
// 93.7 / 101.7, 8192 x 4096 with K = 128 55.4 / 57.5, 192 59.5 / 59.6, 512 96 / 89; three formats K = 64 102.7 / 104.8, 256 113.2 / 119.1,
// 384 131.2 / 131.9, 416 138.0 / 134.7.  A launch that mixes the two takes what its long units want.
bool r_by_warps(bool side, const UnitPlan* units, int n) {
  for (int k = 0; k < n; ++k)
    if (units[k].g.K > (side ? 2 : CfgP::kStages) * kBlockK) return true;
  return false;
}

// What a tile of a unit takes its CTA pair, in cycles: a block of the contraction in all three products 950 in the side-by-side
// form; else 683 for the bf16 products and 430 for 128 entries of each 8-bit one; a tile's fixed part beside that, and
// with short contractions the epilogue's (8192 x 4096, K = 64 ... 4096, whole launches over rounds of tiles).
double tile_cycles(bool side, int64_t K, int n_var) {
  const double kb = (double)((K + kBlockK - 1) / kBlockK), nb = (double)((K + CfgP::kLpDepth - 1) / CfgP::kLpDepth);
  if (side) return std::max(4000.0 + 950.0 * kb, 6000.0);
  return std::max(2500.0 + 683.0 * kb + n_var * (600.0 + 430.0 * nb), 5000.0 + 2700.0 * n_var);
}

// Deals the tiles of a launch's units, in the order of descending cost, to the pairs: each unit's to those with the least to do
// so far.  Where the cheap units have tiles enough to fill what the dear ones leave uneven, the pairs end within a tile of the cheapest
// kind of one another; else within one of the dearest.  (Dealt in rounds of a tile for each pair, the
// four products of a BERT-base layer, 96 tiles of K = 3072 and 768 of 768, took 18 units of the cheap tile where 15.6 would
// do: the launch 176 us, 165 so; a sweep layer's 4.82 ms, 4.58, a BERT-large layer's 2.34, 2.25.)  A pair that has a tile's
// time less to do than another takes its tiles ahead of the rounds (lead), the remainder comes after them (last), so that pairs
// are in the same round and share the blocks they read.  A pair that goes on to another unit has its records to write and the next
// unit's words to fetch, about 4000 cycles: of pairs that would end at the same time, those that have the unit already take its
// rest (two products of 49 and 42 tiles of K = 768 in two formats 32.5 us when they do not, 30.6 so).
struct TileDeal {
  static constexpr double kUnitCycles = 4000.0;
  // neighbouring pairs with the same load and first unit (-1: none yet): a unit splits one run at most, so that it costs the host a tenth of a
  // microsecond
  struct Run { int p0, n; double load; int64_t count; int first; };
  Run runs[2 * kMaxPairs];
  int n_runs = 1, pairs;
  explicit TileDeal(int n) : pairs(n) { runs[0] = Run{0, n, 0.0, 0, -1}; }
  template <typename Key>
  void sort_runs(Key key) {                                // by insertion: a few runs, nearly in order
    for (int i = 1; i < n_runs; ++i) {
      const Run r = runs[i];
      int j = i;
      for (; j > 0 && (key(runs[j - 1]) > key(r) || (key(runs[j - 1]) == key(r) && runs[j - 1].p0 > r.p0)); --j) runs[j] = runs[j - 1];
      runs[j] = r;
    }
  }
  // the first `n` pairs of run i become a run of their own, before it
  void split(int i, int n) {
    for (int j = n_runs++; j > i + 1; --j) runs[j] = runs[j - 1];
    runs[i + 1] = runs[i];
    runs[i + 1].p0 += n; runs[i + 1].n -= n;
    runs[i].n = n;
  }
  void deal(int unit, int64_t tiles, double cost, GroupUnit* u, uint16_t* lead) {
    sort_runs([](const Run& r) { return r.load; });
    // neighbours that have come to the same load are one run again
    int last = 0;
    for (int i = 1; i < n_runs; ++i) {
      if (runs[i].load == runs[last].load && runs[i].first == runs[last].first && runs[i].p0 == runs[last].p0 + runs[last].n) runs[last].n += runs[i].n;
      else runs[++last] = runs[i];
    }
    n_runs = last + 1;
    // the level that the work of all these tiles fills the lowest loads up to, and whole tiles below it
    double level = 0.0, below = 0.0;
    for (int i = 0, width = 0; i < n_runs; ++i) {
      below += runs[i].load * runs[i].n;
      width += runs[i].n;
      level = ((double)tiles * cost + below) / width;
      if (i + 1 == n_runs || level <= runs[i + 1].load) break;
    }
    const double most = runs[n_runs - 1].load, per_cost = 1.0 / cost;
    int64_t left = tiles, rounds = tiles;
    for (int i = 0; i < n_runs; ++i) {
      Run& r = runs[i];
      r.count = level > r.load ? (int64_t)((level - r.load) * per_cost) : 0;
      if (r.count * r.n > left) r.count = left / r.n;
      left -= r.count * r.n;
    }
    // the rest, less than one for each pair, where it ends earliest
    auto changes = [](const Run& r) { return r.load > 0.0 ? kUnitCycles : 0.0; };      // what a unit costs a pair beside its tiles
    sort_runs([&](const Run& r) { return r.load + cost * r.count + (r.count == 0 ? changes(r) : 0.0); });
    for (int i = 0; left > 0; i = i + 1 == n_runs ? 0 : i + 1) {
      if (left < runs[i].n) split(i, (int)left);
      ++runs[i].count;
      left -= runs[i].n;
    }
    for (int i = 0; i < n_runs; ++i) rounds = std::min(rounds, runs[i].count);
    const bool even = tiles - rounds * pairs > 65535;      // beyond the prefix sums' type: dealt evenly
    if (even) {
      rounds = tiles / pairs;
      const int rest = (int)(tiles % pairs);
      for (int i = 0; i < n_runs; ++i)
        if (runs[i].p0 < rest && rest < runs[i].p0 + runs[i].n) split(i, rest - runs[i].p0);
      for (int i = 0; i < n_runs; ++i) runs[i].count = rounds + (runs[i].p0 < rest ? 1 : 0);
    }
    for (uint32_t& w : u->last) w = 0;
    memset(lead, 0, sizeof(uint16_t) * (size_t)(pairs + 1));
    bool any_lead = false;
    for (int i = 0; i < n_runs; ++i) {
      Run& r = runs[i];
      // one of the tiles beside the rounds comes last, unless the pair is that far behind with all of them
      const int64_t more = r.count - rounds;
      const bool one_last = more > 0 && (even || most - r.load < cost * more);
      if (one_last)
        for (int w = r.p0 >> 5, end = r.p0 + r.n; w * 32 < end; ++w) {
          const int lo = std::max(r.p0 - 32 * w, 0), n = std::min(end - 32 * w, 32) - lo;
          u->last[w] |= (n == 32 ? ~0u : (1u << n) - 1u) << lo;
        }
      if (more > one_last) {
        any_lead = true;
        for (int p = r.p0; p < r.p0 + r.n; ++p) lead[p + 1] = (uint16_t)(more - one_last);
      }
      r.load += cost * r.count + (r.count > 0 ? changes(r) : 0.0);
      if (r.first < 0 && r.count > 0) r.first = unit;
    }
    if (any_lead)
      for (int p = 0; p < pairs; ++p) lead[p + 1] = (uint16_t)(lead[p + 1] + lead[p]);
    u->rounds = (int32_t)rounds; u->n_lead = lead[pairs];
  }
  void first_units(uint8_t* first) const {
    for (int i = 0; i < n_runs; ++i) memset(first + runs[i].p0, std::max(runs[i].first, 0), (size_t)runs[i].n);
  }
};

template <bool SIDE, typename Table>
qm_status launch_units(const TcProbeArgs* ps, const UnitPlan* units, int n, bool mn, cudaStream_t s) {
  static Table tab;                    // up to 30 KB: kept off the stack; guarded by the mutex below
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  const TcProbeArgs& first = ps[units[0].probe[0]];
  tab.n = n;
  tab.n_var = 0;
  tab.wait_limit_ns = g_wait_limit_ns.load();
  tab.stop_after_kb = g_stop_after_kb.load();
  tab.done_counter = first.done_counter;
  tab.err0 = first.err_word;
  tab.prepare_flags = first.prepare_flags;
  int64_t total = 0;
  for (int k = 0; k < n; ++k) total += tile_count(units[k].g);
  const int pairs = (int)std::min<int64_t>(total, max_pairs());
  TileDeal pair_loads(pairs);
  for (int k = 0; k < n; ++k) {
    const UnitPlan& up = units[k];
    const GemmShape g = up.g;
    const TcProbeArgs& p0 = ps[up.probe[0]];
    GroupUnit& gu = tab.u[k];
    // outputs at most 64 wide (the context and score-gradient products of attention): MMAs of N = 64,
    // half as many right-operand rows staged
    const int half_n = g.N <= 64 ? 32 : kHalfN;
    // an operand with the contraction strided is staged as it lies in memory: mn-major tiles
    const bool have = (p0.l_mn ? make_map_mn(&tab.unit_maps[k][0], p0.l, true, 64, kBlockK, g.K, g.M, g.batch, p0.l_ld, p0.l_sb)
                                 : make_map(&tab.unit_maps[k][0], p0.l, true, kBlockM, g.K, g.M, g.batch, p0.l_ld, p0.l_sb)) &&
                      (p0.r_mn ? make_map_mn(&tab.unit_maps[k][1], p0.r, true, half_n, kBlockK, g.K, g.N, g.batch, p0.r_ld, p0.r_sb)
                                 : make_map(&tab.unit_maps[k][1], p0.r, true, half_n, g.K, g.N, g.batch, p0.r_ld, p0.r_sb));
    if (!have) return QM_ERR_CUDA;
    gu.major = (p0.l_mn ? kUnitMnMajorL : 0u) | (p0.r_mn ? kUnitMnMajorR : 0u);
    KernelArgs ka{};
    fill_tiles(&ka, g);
    gu.M = (int32_t)g.M; gu.N = (int32_t)g.N; gu.K = (int32_t)g.K;
    gu.tiles_m = ka.tiles_m; gu.tiles_n = ka.tiles_n;
    pair_loads.deal(k, ka.num_tiles, up.cycles, &gu, tab.lead[k]);
    gu.half_n = half_n;
    // Tiles that run at the same time should share the LARGER operand's blocks, so that it is
    // streamed from HBM once and the smaller one is what gets fetched again (from L2, if it fits):
    // the tiles of a batch element are walked along the shorter side first.
    gu.m_fastest = g.M < g.N ? 1 : 0;
    const Divisor by_b((uint32_t)(gu.tiles_m * gu.tiles_n)), by_inner((uint32_t)(gu.m_fastest ? gu.tiles_m : gu.tiles_n));
    gu.b_mul = by_b.mul; gu.b_shift = (uint8_t)by_b.shift; gu.i_mul = by_inner.mul; gu.i_shift = (uint8_t)by_inner.shift;
    gu.var_begin = (int16_t)tab.n_var; gu.n_var = (int16_t)up.n_var;
    for (int j = 0; j < up.n_var; ++j) {
      const TcProbeArgs& p = ps[up.probe[j]];
      if (Table::kUnits != 1 && p.prepare_flags) return QM_ERR_UNSUPPORTED;      // read for probes that are launched alone only
      CUtensorMap(&vm)[2] = tab.var_maps[tab.n_var];
      VarInfo& info = tab.info[tab.n_var];
      tab.count[tab.n_var] = (uint64_t)(g.M * g.N * g.batch);
      GroupVar& v = tab.v[tab.n_var++];
      // blocks of codes are 64 entries deep beside the bf16 tiles, 128 on their own
      const int depth = SIDE ? kBlockK : CfgP::kLpDepth;
      auto code_map = [&](CUtensorMap* m, const uint8_t* codes, bool mn, int box_rows, int64_t rows) {
        const int64_t ld = qm_code_ld(mn ? rows : g.K);
        return mn ? make_map_mn(m, codes, false, box_rows, depth, g.K, rows, g.batch, ld, g.K * ld)
                           : make_map(m, codes, false, box_rows, g.K, rows, g.batch, ld, rows * ld, !SIDE);
      };
      if (!code_map(&vm[0], p.cl, p.cl_mn, kBlockM, g.M) || !code_map(&vm[1], p.cr, p.cr_mn, half_n, g.N)) return QM_ERR_CUDA;
      v.dl = p.dl; v.dr = p.dr;
      v.partials = p.partials; v.result = p.result; v.row_stats = p.row_stats;
      v.err_word = p.err_word; v.err_also[0] = p.err_also[0]; v.err_also[1] = p.err_also[1];
      info.flags = (p.fmt_l == QM_FMT_INT8 ? kVarI8 : 0u) | (p.gran_l == QM_GRAN_CHANNEL ? kVarScalePerRow : 0u) |
                (p.gran_r == QM_GRAN_CHANNEL ? kVarScalePerCol : 0u) | (p.row_stats ? kVarRowStats : 0u) |
                (p.cl_mn ? kVarMnMajorL : 0u) | (p.cr_mn ? kVarMnMajorR : 0u);
      info.idesc = lp_idesc(p.fmt_l, p.fmt_r, 2 * half_n) | (p.cl_mn ? kIdescMnMajorA : 0u) | (p.cr_mn ? kIdescMnMajorB : 0u);
    }
  }
  pair_loads.first_units(tab.first);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(2 * pairs));
  cfg.blockDim = dim3(kProbeThreads);
  cfg.dynamicSmemBytes = ProbeKernel<SIDE, false, false, Table>::kSmem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 2 : 1;
  const bool rw = r_by_warps(SIDE, units, n);
  const auto kernel = mn ? (rw ? ProbeKernel<SIDE, true, true, Table>::kernel : ProbeKernel<SIDE, true, false, Table>::kernel)
                         : (rw ? ProbeKernel<SIDE, false, true, Table>::kernel : ProbeKernel<SIDE, false, false, Table>::kernel);
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  profile_events(&ev0, &ev1);
  if (ev0) QM_CUDA_OK(cudaEventRecord(ev0, s));
  QM_CUDA_OK(cudaLaunchKernelEx(&cfg, kernel, tab));
  if (ev1) QM_CUDA_OK(cudaEventRecord(ev1, s));
  count_launch();
  return QM_OK;
}
}  // namespace

void set_wait_limit_ns(uint64_t ns) { g_wait_limit_ns.store(ns ? ns : 1000000000ull); }
void set_stop_after_kb(uint32_t kb) { g_stop_after_kb.store(kb); }

qm_status launch_tc_probes(const TcProbeArgs* ps, int n, cudaStream_t s) {
  if (n < 1) return QM_ERR_INVALID_ARG;
  qm_status st = probe_residency();
  if (st != QM_OK) return st;
  // units: probes of the same operands, up to the first probe whose extents are refused
  std::vector<UnitPlan> units;
  units.reserve((size_t)n);
  qm_status refused = QM_OK;
  for (int i = 0; i < n; ++i) {
    if (!shape_ok(ps[i].g) || ps[i].cl2) { refused = QM_ERR_UNSUPPORTED; break; }
    UnitPlan* u = nullptr;
    for (UnitPlan& c : units)
      if (c.n_var < kMaxVar && same_products(ps[c.probe[0]], ps[i])) { u = &c; break; }
    if (!u) {
      units.push_back(UnitPlan{ps[i].g, 0, {}, 0.0});
      u = &units.back();
    }
    u->probe[u->n_var++] = i;
  }
  // Units of one probe go to the side-by-side kernel, ahead of the others, unless they could not fill the GPU and there
  // are others: a launch more costs its set-up and drain, about 10 us, and they ride along instead.
  auto single = [](const UnitPlan& u) { return u.n_var == 1; };
  const auto others = std::stable_partition(units.begin(), units.end(), single);
  int64_t single_tiles = 0;
  for (auto u = units.begin(); u != others; ++u) single_tiles += tile_count(u->g);
  const size_t n_side = others == units.end() || single_tiles >= max_pairs() ? (size_t)(others - units.begin()) : 0;
  for (size_t k = 0; k < units.size(); ++k) units[k].cycles = tile_cycles(k < n_side, units[k].g.K, units[k].n_var);
  auto by_cost = [](const UnitPlan& a, const UnitPlan& b) { return a.cycles > b.cycles; };      // descending
  std::stable_sort(units.begin(), units.begin() + n_side, by_cost);
  std::stable_sort(units.begin() + n_side, units.end(), by_cost);
  auto any_mn = [&](const UnitPlan* u, int count) {
    for (int k = 0; k < count; ++k) {
      const TcProbeArgs& a = ps[u[k].probe[0]];
      if (a.l_mn || a.r_mn || a.cl_mn || a.cr_mn) return true;
    }
    return false;
  };
  for (size_t u0 = 0; u0 < units.size() && st == QM_OK;) {
    const bool side = u0 < n_side;
    const size_t end = side ? n_side : units.size();
    size_t u1 = u0;
    int64_t tiles = 0;
    int vars = 0;
    while (u1 < end && (int)(u1 - u0) < TableBig::kUnits && vars + units[u1].n_var <= TableBig::kVars &&
           tiles + tile_count(units[u1].g) < (1ll << 31)) {
      vars += units[u1].n_var;
      tiles += tile_count(units[u1].g);
      ++u1;
    }
    const int count = (int)(u1 - u0);
    const bool mn = any_mn(&units[u0], count);
    if (!side) st = launch_units<false, TableBig>(ps, &units[u0], count, mn, s);
    else if (count == 1) st = launch_units<true, TableOne>(ps, &units[u0], 1, mn, s);
    else st = launch_units<true, TableBig>(ps, &units[u0], count, mn, s);
    u0 = u1;
  }
  return st != QM_OK ? st : refused;
}

// per format; a launch writes one record per CTA of its grid
int tc_probe_records(GemmShape) {
  (void)probe_residency();
  return 2 * max_pairs();
}

qm_status launch_tc_probe(const TcProbeArgs& p, cudaStream_t s) {
  if (!p.cl2) return launch_tc_probes(&p, 1, s);            // one format: a unit of one
  if (!shape_ok(p.g)) return QM_ERR_UNSUPPORTED;
  const qm_status rs = probe_residency();
  if (rs != QM_OK) return rs;
  const GemmShape g = p.g;
  const int64_t ldc = qm_code_ld(g.K);
  CUtensorMap maps[8];
  bool ok = make_map(&maps[0], p.l, true, kBlockM, g.K, g.M, g.batch, p.l_ld, p.l_sb) &&
            make_map(&maps[1], p.r, true, kHalfN, g.K, g.N, g.batch, p.r_ld, p.r_sb) &&
            make_map(&maps[2], p.l_abs, true, kBlockM, g.K, g.M, g.batch, g.K, g.M * g.K) &&
            make_map(&maps[3], p.r_abs, true, kHalfN, g.K, g.N, g.batch, g.K, g.N * g.K) &&
            make_map(&maps[4], p.cl, false, kBlockM, g.K, g.M, g.batch, ldc, g.M * ldc) &&
            make_map(&maps[5], p.cr, false, kHalfN, g.K, g.N, g.batch, ldc, g.N * ldc) &&
            make_map(&maps[6], p.cl2, false, kBlockM, g.K, g.M, g.batch, ldc, g.M * ldc) &&
            make_map(&maps[7], p.cr2, false, kHalfN, g.K, g.N, g.batch, ldc, g.N * ldc);
  if (!ok) return QM_ERR_CUDA;
  KernelArgs ka{};
  fill_tiles(&ka, g);
  ka.dl = p.dl; ka.pc_l = p.gran_l == QM_GRAN_CHANNEL; ka.dr = p.dr; ka.pc_r = p.gran_r == QM_GRAN_CHANNEL;
  ka.partials = p.partials; ka.done_counter = p.done_counter; ka.result = p.result;
  ka.count = (uint64_t)(g.M * g.N * g.batch);
  ka.err_word = p.err_word; ka.idesc_lp = lp_idesc(p.fmt_l, p.fmt_r);
  // the first format is an FP8 one (the caller orders them), the second FP8 or INT8
  if (p.fmt_l == QM_FMT_INT8) return QM_ERR_UNSUPPORTED;
  ka.dl2 = p.dl2; ka.dr2 = p.dr2; ka.idesc_lp2 = lp_idesc(p.fmt_l2, p.fmt_r2);
  return p.fmt_l2 == QM_FMT_INT8 ? launch<kProbe2, kKindF8, kKindI8>(maps, ka, g, s)
                                 : launch<kProbe2, kKindF8, kKindF8>(maps, ka, g, s);
}

qm_status launch_tc_gemm_lp(const uint8_t* cl, int fmt_l, const float* dl, int gran_l,
                            const uint8_t* cr, int fmt_r, const float* dr, int gran_r, GemmShape g,
                            float* out_descaled, void* out_raw, uint32_t* err_word, cudaStream_t s) {
  if (!shape_ok(g)) return QM_ERR_UNSUPPORTED;
  const int64_t ldc = qm_code_ld(g.K);
  CUtensorMap maps[8];
  if (use_wide(g)) {
    if (!make_map(&maps[0], cl, false, kBlockM, g.K, g.M, g.batch, ldc, g.M * ldc, true) ||
        !make_map(&maps[1], cr, false, kWideHalfN, g.K, g.N, g.batch, ldc, g.N * ldc, true))
      return QM_ERR_CUDA;
    KernelArgs kw{};
    kw.M = g.M; kw.N = g.N; kw.K = g.K;
    kw.dl = dl; kw.pc_l = gran_l == QM_GRAN_CHANNEL; kw.dr = dr; kw.pc_r = gran_r == QM_GRAN_CHANNEL;
    kw.out_descaled = out_descaled; kw.out_raw = out_raw; kw.err_word = err_word;
    const uint32_t fa = fmt_l == QM_FMT_E4M3 ? 0u : 1u, fb = fmt_r == QM_FMT_E4M3 ? 0u : 1u;
    kw.idesc_lp = fmt_l == QM_FMT_INT8 ? make_idesc(2, 1, 1, kPairM, kWideN) : make_idesc(1, fa, fb, kPairM, kWideN);
    return fmt_l == QM_FMT_INT8 ? launch_wide<kKindI8>(maps[0], maps[1], kw, g, s)
                                : launch_wide<kKindF8>(maps[0], maps[1], kw, g, s);
  }
  bool ok = make_map(&maps[4], cl, false, kBlockM, g.K, g.M, g.batch, ldc, g.M * ldc) &&
            make_map(&maps[5], cr, false, kHalfN, g.K, g.N, g.batch, ldc, g.N * ldc);
  if (!ok) return QM_ERR_CUDA;
  maps[0] = maps[1] = maps[2] = maps[3] = maps[6] = maps[7] = maps[4];
  KernelArgs ka{};
  fill_tiles(&ka, g);
  ka.dl = dl; ka.pc_l = gran_l == QM_GRAN_CHANNEL; ka.dr = dr; ka.pc_r = gran_r == QM_GRAN_CHANNEL;
  ka.out_descaled = out_descaled; ka.out_raw = out_raw; ka.err_word = err_word;
  ka.idesc_lp = lp_idesc(fmt_l, fmt_r);
  return fmt_l == QM_FMT_INT8 ? launch<kLpOnly, kKindI8>(maps, ka, g, s)
                              : launch<kLpOnly, kKindF8>(maps, ka, g, s);
}

qm_status launch_tc_gemm_ref(const void* l, const void* r, GemmShape g, float* out, uint32_t* err_word,
                             cudaStream_t s) {
  if (!shape_ok(g)) return QM_ERR_UNSUPPORTED;
  CUtensorMap maps[8];
  if (use_wide(g)) {
    if (!make_map(&maps[0], l, true, kBlockM, g.K, g.M, g.batch, g.K, g.M * g.K, true) ||
        !make_map(&maps[1], r, true, kWideHalfN, g.K, g.N, g.batch, g.K, g.N * g.K, true))
      return QM_ERR_CUDA;
    KernelArgs kw{};
    kw.M = g.M; kw.N = g.N; kw.K = g.K;
    kw.out_descaled = out; kw.err_word = err_word;
    return launch_wide<kKindF16>(maps[0], maps[1], kw, g, s);
  }
  bool ok = make_map(&maps[0], l, true, kBlockM, g.K, g.M, g.batch, g.K, g.M * g.K) &&
            make_map(&maps[1], r, true, kHalfN, g.K, g.N, g.batch, g.K, g.N * g.K);
  if (!ok) return QM_ERR_CUDA;
  maps[2] = maps[3] = maps[4] = maps[5] = maps[6] = maps[7] = maps[0];
  KernelArgs ka{};
  fill_tiles(&ka, g);
  ka.out_descaled = out; ka.err_word = err_word;
  return launch<kRefOnly, kKindF8>(maps, ka, g, s);
}

}  // namespace qm
