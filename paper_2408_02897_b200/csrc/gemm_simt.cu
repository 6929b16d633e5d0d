// CUDA-core versions of the probe's products.  They serve the fp32-reference configuration
// (fp32 operands have no tensor-core path with an fp32 multiply) and act as a second opinion
// for the tensor-core kernels in the tests.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "qm_internal.h"
#include "reduce.cuh"

namespace qm {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ float decode_code(uint32_t c, int fmt) {
  uint32_t h2;
  uint16_t in = (uint16_t)(c & 0xffu);
  if (fmt == QM_FMT_E4M3) asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"(in));
  else asm("cvt.rn.f16x2.e5m2x2 %0, %1;" : "=r"(h2) : "h"(in));
  __half lo = __ushort_as_half((unsigned short)(h2 & 0xffffu));
  return __half2float(lo);
}

struct SimtOperand {
  const void* p; int dtype;               // the unquantized operand (probe only)
  int64_t rows, s_nc, s_c, s_b;
  const uint8_t* codes; int fmt;
  const float* delta; int per_channel;
};
struct SimtArgs {
  SimtOperand l, r;
  int64_t K, ldc;
  float* out_descaled; void* out_raw;                       // plain product
  double* partials; uint32_t* done_counter;                 // probe: a record per block; counts finished blocks
  uint32_t* err_word; const uint32_t* prepare_flags; qm_metric_result* result; uint64_t count;
};

// A block computes a TM x TN output tile with 256 threads, 4 x 4 outputs each.  The work is fp32 FMA (three
// per output and contraction entry); what bounds small products is that a 64 x 64 tiling gives them a
// handful of blocks that walk the whole contraction alone.  So there are four tile shapes, and where a
// tile needs fewer than 256 threads the rest split the contraction: SPLIT groups of T threads take KG
// consecutive entries each of every chunk of KC, and their accumulators are added through shared memory
// at the end (a fixed order).  A chunk of all four matrices is fetched into registers with
// 16-byte loads while the previous one is being multiplied and stored to the other half of shared memory.
template <int TM, int TN>
struct Tile {
  static constexpr int T = (TM / 4) * (TN / 4), SPLIT = kThreads / T;
  static constexpr int KG = SPLIT == 1 ? 32 : 16, KC = KG * SPLIT;
  static constexpr size_t kStage = (size_t)KC * (TM + TN) * 2;              // floats: both operands, values and codes
  static constexpr size_t kReduce = SPLIT > 1 ? (size_t)kThreads * 48 : 0;
  static constexpr size_t kSmem = 4 * (2 * kStage > kReduce ? 2 * kStage : kReduce);
};

// [k][row] matrices in shared memory, rows in units of four that are permuted with k: the transposing
// stores of a contraction-contiguous operand and the 16-byte reads of the main loop both spread over the banks.
template <int ROWS>
__device__ __forceinline__ int slot4(int k, int unit) { return k * ROWS + ((unit ^ ((k >> 2) & (ROWS / 4 - 1))) << 2); }

template <int ROWS, int KC>
struct Fetch {
  static constexpr int NV = ROWS * KC / 4 / kThreads;         // vectors of four elements per thread
  float4 v[NV];
  uint32_t c[NV];
  bool along_k;

  static __device__ __forceinline__ float get1(const SimtOperand& o, int64_t off) {
    if (o.dtype == QM_DT_BF16)
      return __uint_as_float((uint32_t)__ldg(reinterpret_cast<const unsigned short*>(o.p) + off) << 16);
    return __ldg(reinterpret_cast<const float*>(o.p) + off);
  }
  // four elements along the contiguous dimension, `left` of which exist; views start on 16 bytes and their
  // other stride is a multiple of eight elements, so whole vectors are aligned
  static __device__ __forceinline__ float4 get4(const SimtOperand& o, int64_t off, int64_t left) {
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (left >= 4) {
      if (o.dtype == QM_DT_BF16) {
        const uint2 w = __ldg(reinterpret_cast<const uint2*>(reinterpret_cast<const unsigned short*>(o.p) + off));
        x.x = __uint_as_float(w.x << 16); x.y = __uint_as_float(w.x & 0xffff0000u);
        x.z = __uint_as_float(w.y << 16); x.w = __uint_as_float(w.y & 0xffff0000u);
      } else {
        x = __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(o.p) + off));
      }
    } else if (left > 0) {
      x.x = get1(o, off);
      if (left > 1) x.y = get1(o, off + 1);
      if (left > 2) x.z = get1(o, off + 2);
    }
    return x;
  }
  template <bool VALUES>
  __device__ __forceinline__ void load(const SimtOperand& o, int64_t b, int64_t row0, int64_t k0, int64_t K, int64_t ldc) {
    along_k = o.s_c == 1;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int t = threadIdx.x + i * kThreads;
      const int64_t row = row0 + t / (KC / 4), k = k0 + 4 * (t % (KC / 4));
      // rows of codes are a multiple of 16 long, zero beyond K where the probe made them
      c[i] = row < o.rows && k < ldc ? __ldg(reinterpret_cast<const uint32_t*>(o.codes + (b * o.rows + row) * ldc + k)) : 0u;
      if (!VALUES) continue;
      if (along_k) {
        v[i] = get4(o, b * o.s_b + row * o.s_nc + k, row < o.rows ? K - k : 0);
      } else {
        const int64_t r4 = row0 + 4 * (t % (ROWS / 4)), kk = k0 + t / (ROWS / 4);
        v[i] = get4(o, b * o.s_b + kk * o.s_c + r4, kk < K ? o.rows - r4 : 0);
      }
    }
    // a caller's codes (plain product) count as zero beyond K, whatever their padding holds
    if (!VALUES && k0 + KC > K) {
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const int64_t left = K - (k0 + 4 * ((threadIdx.x + i * kThreads) % (KC / 4)));
        if (left < 4) c[i] &= left > 0 ? (1u << (8 * (int)left)) - 1u : 0u;
      }
    }
  }
  // values: [KC][ROWS] floats; codes: the same as floats, or [KC / 4][ROWS] words of four bytes (IS_INT)
  template <bool VALUES, bool IS_INT>
  __device__ __forceinline__ void store(float* sv, float* sc, int fmt) const {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int t = threadIdx.x + i * kThreads;
      const int row = t / (KC / 4), k4 = t % (KC / 4);
      if (IS_INT) {
        reinterpret_cast<uint32_t*>(sc)[k4 * ROWS + (((row >> 2) ^ (k4 & (ROWS / 4 - 1))) << 2) + (row & 3)] = c[i];
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) sc[slot4<ROWS>(4 * k4 + j, row >> 2) + (row & 3)] = decode_code(c[i] >> (8 * j), fmt);
      }
      if (!VALUES) continue;
      if (along_k) {
        const float x[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
        for (int j = 0; j < 4; ++j) sv[slot4<ROWS>(4 * k4 + j, row >> 2) + (row & 3)] = x[j];
      } else {
        *reinterpret_cast<float4*>(sv + slot4<ROWS>(t / (ROWS / 4), t % (ROWS / 4))) = v[i];
      }
    }
  }
};

__device__ __forceinline__ void unpack4(float (&x)[4], const float* p) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
}

// PROBE: three accumulators (reference, denominator, 8-bit) and the Eq. 3 partial sums.
// otherwise: the 8-bit product only, written out.
template <bool IS_INT, bool PROBE, int TM, int TN>
__global__ void __launch_bounds__(kThreads, 2) simt_kernel(const SimtArgs a) {
  using C = Tile<TM, TN>;
  constexpr int T = C::T, SPLIT = C::SPLIT, KG = C::KG, KC = C::KC;
  extern __shared__ float4 smem4[];
  float* const smem = reinterpret_cast<float*>(smem4);
  __shared__ double sred[5][8], tot[5];
  __shared__ uint32_t s_last;
  pdl_prologue();
  const int64_t b = blockIdx.z;
  const int64_t m0 = (int64_t)blockIdx.y * TM, n0 = (int64_t)blockIdx.x * TN;
  const int g = threadIdx.x / T, t = threadIdx.x % T;         // group along the contraction, thread of the tile
  const int tx = t % (TN / 4), ty = t / (TN / 4);

  float accC[4][4], accD[4][4], accF[4][4];
  int accI[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) { accC[i][j] = 0.f; accD[i][j] = 0.f; accF[i][j] = 0.f; accI[i][j] = 0; }

  Fetch<TM, KC> fl;
  Fetch<TN, KC> fr;
  fl.template load<PROBE>(a.l, b, m0, 0, a.K, a.ldc);
  fr.template load<PROBE>(a.r, b, n0, 0, a.K, a.ldc);
  int buf = 0;
  for (int64_t k0 = 0; k0 < a.K; k0 += KC, buf ^= 1) {
    float* const sL = smem + buf * C::kStage;
    float* const sR = sL + KC * TM;
    float* const sLq = sR + KC * TN;
    float* const sRq = sLq + KC * TM;
    fl.template store<PROBE, IS_INT>(sL, sLq, a.l.fmt);
    fr.template store<PROBE, IS_INT>(sR, sRq, a.r.fmt);
    __syncthreads();                       // (also: everyone is through with the other half of shared memory)
    if (k0 + KC < a.K) {
      fl.template load<PROBE>(a.l, b, m0, k0 + KC, a.K, a.ldc);
      fr.template load<PROBE>(a.r, b, n0, k0 + KC, a.K, a.ldc);
    }
#pragma unroll 4
    for (int kk = 0; kk < KG; ++kk) {
      const int k = g * KG + kk;
      if (PROBE) {
        float lv[4], rv[4];
        unpack4(lv, sL + slot4<TM>(k, ty));
        unpack4(rv, sR + slot4<TN>(k, tx));
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            accC[i][j] = fmaf(lv[i], rv[j], accC[i][j]);
            accD[i][j] = fmaf(fabsf(lv[i]), fabsf(rv[j]), accD[i][j]);
          }
      }
      if (!IS_INT) {
        float lq[4], rq[4];
        unpack4(lq, sLq + slot4<TM>(k, ty));
        unpack4(rq, sRq + slot4<TN>(k, tx));
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) accF[i][j] = fmaf(lq[i], rq[j], accF[i][j]);
      } else if ((kk & 3) == 0) {          // four entries at once
        const int k4 = k >> 2;
        const int4 lw = *reinterpret_cast<const int4*>(sLq + k4 * TM + ((ty ^ (k4 & (TM / 4 - 1))) << 2));
        const int4 rw = *reinterpret_cast<const int4*>(sRq + k4 * TN + ((tx ^ (k4 & (TN / 4 - 1))) << 2));
        const int lq[4] = {lw.x, lw.y, lw.z, lw.w}, rq[4] = {rw.x, rw.y, rw.z, rw.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) accI[i][j] = __dp4a(lq[i], rq[j], accI[i][j]);
      }
    }
  }

  // outputs of this thread: all 16 of its tile position, or 16 / SPLIT of them once the groups' sums are added
  constexpr int OUT = 16 / SPLIT;
  float vC[OUT], vD[OUT], vF[OUT];
  int vI[OUT];
  if (SPLIT > 1) {
    __syncthreads();                       // the tiles' memory becomes [48][SPLIT][T] accumulators
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      if (PROBE) {
        smem[(e * SPLIT + g) * T + t] = accC[e / 4][e % 4];
        smem[((16 + e) * SPLIT + g) * T + t] = accD[e / 4][e % 4];
      }
      smem[((32 + e) * SPLIT + g) * T + t] = IS_INT ? __int_as_float(accI[e / 4][e % 4]) : accF[e / 4][e % 4];
    }
    __syncthreads();
#pragma unroll
    for (int o = 0; o < OUT; ++o) {
      const int e = g * OUT + o;
      vC[o] = vD[o] = vF[o] = 0.f;
      vI[o] = 0;
#pragma unroll
      for (int h = 0; h < SPLIT; ++h) {
        if (PROBE) {
          vC[o] += smem[(e * SPLIT + h) * T + t];
          vD[o] += smem[((16 + e) * SPLIT + h) * T + t];
        }
        const float f = smem[((32 + e) * SPLIT + h) * T + t];
        if (IS_INT) vI[o] += __float_as_int(f);
        else vF[o] += f;
      }
    }
  } else {
#pragma unroll
    for (int o = 0; o < OUT; ++o) {
      vC[o] = accC[o / 4][o % 4]; vD[o] = accD[o / 4][o % 4]; vF[o] = accF[o / 4][o % 4]; vI[o] = accI[o / 4][o % 4];
    }
  }

  const float dl_t = a.l.per_channel ? 0.f : __ldg(a.l.delta), dr_t = a.r.per_channel ? 0.f : __ldg(a.r.delta);
  float fbe = 0, fmx = 0, fd2 = 0, fr2 = 0, fn2 = 0;
#pragma unroll
  for (int o = 0; o < OUT; ++o) {
    const int e = SPLIT > 1 ? g * OUT + o : o;
    const int64_t mi = m0 + ty * 4 + (e >> 2), ni = n0 + tx * 4 + (e & 3);
    if (mi >= a.l.rows || ni >= a.r.rows) continue;
    const float dl = a.l.per_channel ? __ldg(a.l.delta + b * a.l.rows + mi) : dl_t;
    const float dr = a.r.per_channel ? __ldg(a.r.delta + b * a.r.rows + ni) : dr_t;
    const float acc = IS_INT ? (float)vI[o] : vF[o];
    const float q = acc * (dl * dr);
    if (PROBE) {
      const float c = vC[o], d = vD[o];
      const float diff = c - q;
      const float be = d != 0.f ? __fdiv_rn(fabsf(diff), d) : 0.f;
      fbe += be; fmx = fmaxf(fmx, be);
      fd2 = fmaf(diff, diff, fd2); fr2 = fmaf(c, c, fr2); fn2 = fmaf(d, d, fn2);
    } else {
      const int64_t at = (b * a.l.rows + mi) * a.r.rows + ni;
      if (a.out_descaled) a.out_descaled[at] = q;
      if (a.out_raw) {
        if (IS_INT) reinterpret_cast<int*>(a.out_raw)[at] = vI[o];
        else reinterpret_cast<float*>(a.out_raw)[at] = vF[o];
      }
    }
  }
  if (PROBE) {
    // (the asm keeps what follows of it from being computed ahead of the products and held through them: 72 bytes of spills at 64 x 64, 40 so)
    uint32_t t = threadIdx.x;
    asm volatile("" : "+r"(t));
    double v[4] = {fbe, fd2, fr2, fn2};
    // field of the record that this thread and its seven neighbours hold: the sums around the maximum
    const int held = t >> 3, field = held == 0 ? 0 : held == 4 ? 1 : held + 1;
    const bool writer = (t & 7) == 0 && held < 5;
    double x = block_record<4>(v, fmx, sred, t);
    const int64_t n_blocks = (int64_t)gridDim.x * gridDim.y * gridDim.z;
    const int64_t blk = ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    if (writer) __stcg(a.partials + blk * kPartialDoubles + field, x);
    __syncthreads();
    if (t == 0) {
      __threadfence();                     // after the barrier: covers what the others have written
      s_last = atomicAdd(a.done_counter, 1u) == (uint32_t)(n_blocks - 1) ? 1u : 0u;
    }
    __syncthreads();
    if (s_last) {                          // the last block adds all records up, in a fixed order
      __threadfence();
      v[0] = v[1] = v[2] = v[3] = 0.0;
      float mx = 0.f;
      for (int64_t k = t; k < n_blocks; k += kThreads) {
        const double* rec = a.partials + k * kPartialDoubles;
        v[0] += __ldcg(rec); mx = fmaxf(mx, (float)__ldcg(rec + 1)); v[1] += __ldcg(rec + 2);
        v[2] += __ldcg(rec + 3); v[3] += __ldcg(rec + 4);
      }
      const int not_finite = __syncthreads_or(a.prepare_flags && t < kPrepareFlagWords && __ldcg(a.prepare_flags + t));
      x = block_record<4>(v, mx, sred, t);
      if (writer) tot[field] = x;
      __syncthreads();
      if (t == 0) {                // (the record may be in host memory: stores only, every field once)
        a.result->sum_be = tot[0]; a.result->max_be = tot[1]; a.result->sum_diff2 = tot[2];
        a.result->sum_ref2 = tot[3]; a.result->sum_den2 = tot[4];
        a.result->count = a.count;
        a.result->device_error = *reinterpret_cast<volatile uint32_t*>(a.err_word) | (not_finite ? QM_DEVERR_NONFINITE : 0u);
        a.result->reserved = 0;
      }
    }
  }
}

// The shape whose busiest SM is through first: the blocks there, times what a block takes (fitted: a 32 x 32 block 1.3 times its share of
// a 64 x 64 one, a 16 x 32 block 1.75 times), over the rate at which one block (0.62 of the issue slots) or several (0.85) issue.
// What this is for: a few blocks more than the GPU has SMs double the time.  Contractions below 96 are bound as much by what a block does
// once, and take the largest shape with five blocks for four SMs, those below 64 the largest with more blocks than SMs.  64 x 64 / 32 x 64, us: 640 x 960 (150
// blocks of 64 x 64) K = 20 17.5 / 18.3, 60 23.7 / 23.7, 80 30.5 / 29.3, 95 30.9 / 30.0; 900 x 900 (225) K = 20 17.8 / 20.6, 80 30.9 / 30.5, 95 31.3 / 32.7; 1200 x 800
// (247) K = 95 33.0 / 36.0; 690 x 307 x 65 INT8 220 blocks of 32 x 32 19.8, 440 of 16 x 32 22.1; 900 x 900 x 120 35.1 / 34.1.  Whole probes of 700 x 400 x 368: 154 blocks of 32 x 64 53.7 us, 286 of 32 x 32 37.2; 1024^3 64 x 64
// 205, 32 x 32 232; 400 x 400 x 300 INT8 32 x 32 28.4, 16 x 32 35.8; 128 x 256 x 256 64 blocks of 16 x 32.
constexpr int kShapes[4][2] = {{64, 64}, {32, 64}, {32, 32}, {16, 32}};
dim3 grid_of(GemmShape g, int shape) {
  const int tm = kShapes[shape][0], tn = kShapes[shape][1];
  return dim3((unsigned)((g.N + tn - 1) / tn), (unsigned)((g.M + tm - 1) / tm), (unsigned)g.batch);
}
int shape_of(GemmShape g) {
  constexpr double kBlockCost[4] = {4096.0, 2212.0, 1331.0, 900.0};
  int best = 0;
  double least = 0.0;
  for (int i = 0; i < 4; ++i) {
    const int64_t tm = kShapes[i][0], tn = kShapes[i][1], rows = (g.M + tm - 1) / tm;
    if (i > 0 && rows > 65535) break;                 // (the limit of the grid holds for the largest shape only)
    const int64_t blocks = rows * ((g.N + tn - 1) / tn) * g.batch, sms = sm_count(), per_sm = (blocks + sms - 1) / sms;
    if (g.K < 64 ? blocks > sms : g.K < 96 && i < 3 && 4 * blocks >= 5 * sms) return i;
    const double cost = (double)per_sm * kBlockCost[i] / (per_sm == 1 ? 0.62 : 0.85);
    if (i == 0 || cost < least) { best = i; least = cost; }
  }
  return best;
}

template <bool IS_INT, bool PROBE, int TM, int TN>
qm_status launch_tile(const SimtArgs& a, dim3 grid, cudaStream_t s) {
  constexpr size_t smem = Tile<TM, TN>::kSmem;
  static bool attr_done[kMaxDevices] = {};
  const int dev = current_device();
  if (dev < 0) return QM_ERR_UNSUPPORTED;
  if (!attr_done[dev]) {
    QM_CUDA_OK(cudaFuncSetAttribute(simt_kernel<IS_INT, PROBE, TM, TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    attr_done[dev] = true;
  }
  QM_CUDA_OK(launch_pdl(simt_kernel<IS_INT, PROBE, TM, TN>, grid, dim3(kThreads), smem, s, a));
  count_launch();
  return QM_OK;
}

template <bool PROBE>
qm_status launch_simt(const SimtArgs& a, GemmShape g, cudaStream_t s) {
  const int shape = shape_of(g);
  const dim3 grid = grid_of(g, shape);
  // (64 x 64 tiles, the limits of the grid: what is accepted does not depend on the shape taken)
  if (g.batch > 65535 || (g.M + 63) / 64 > 65535 || grid.y > 65535) return QM_ERR_UNSUPPORTED;
#define QM_S(TM, TN) (a.l.fmt == QM_FMT_INT8 ? launch_tile<true, PROBE, TM, TN>(a, grid, s) : launch_tile<false, PROBE, TM, TN>(a, grid, s))
  switch (shape) {
    case 0: return QM_S(64, 64);
    case 1: return QM_S(32, 64);
    case 2: return QM_S(32, 32);
    default: return QM_S(16, 32);
  }
#undef QM_S
}

}  // namespace

int simt_probe_blocks(GemmShape g) {
  dim3 d = grid_of(g, shape_of(g));
  return (int)(d.x * d.y * d.z);
}

qm_status launch_simt_gemm_lp(const uint8_t* cl, int fmt_l, const float* dl, int gran_l,
                              const uint8_t* cr, int fmt_r, const float* dr, int gran_r,
                              GemmShape g, float* out_descaled, void* out_raw, cudaStream_t s) {
  SimtArgs a{};
  a.l.rows = g.M; a.l.codes = cl; a.l.fmt = fmt_l; a.l.delta = dl; a.l.per_channel = gran_l == QM_GRAN_CHANNEL;
  a.r.rows = g.N; a.r.codes = cr; a.r.fmt = fmt_r; a.r.delta = dr; a.r.per_channel = gran_r == QM_GRAN_CHANNEL;
  a.K = g.K; a.ldc = qm_code_ld(g.K); a.out_descaled = out_descaled; a.out_raw = out_raw;
  return launch_simt<false>(a, g, s);
}

qm_status launch_simt_probe(const View& L, const View& R, const uint8_t* cl, int fmt_l,
                            const float* dl, int gran_l, const uint8_t* cr, int fmt_r,
                            const float* dr, int gran_r, double* partials, uint32_t* done_counter,
                            uint32_t* err_word, const uint32_t* prepare_flags, qm_metric_result* out, cudaStream_t s) {
  GemmShape g{L.nc, R.nc, L.c, L.batch};
  SimtArgs a{};
  a.l = SimtOperand{L.data, L.dtype, L.nc, L.s_nc, L.s_c, L.s_b, cl, fmt_l, dl, gran_l == QM_GRAN_CHANNEL};
  a.r = SimtOperand{R.data, R.dtype, R.nc, R.s_nc, R.s_c, R.s_b, cr, fmt_r, dr, gran_r == QM_GRAN_CHANNEL};
  a.K = L.c; a.ldc = qm_code_ld(L.c); a.partials = partials; a.done_counter = done_counter; a.err_word = err_word; a.prepare_flags = prepare_flags;
  a.result = out; a.count = (uint64_t)(g.M * g.N * g.batch);
  return launch_simt<true>(a, g, s);
}

}  // namespace qm
