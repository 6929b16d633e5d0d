// Scale (Eq. 1, right half) and quantize (Eq. 1, left half + saturation rule) kernels.
// All of them are HBM-bound streaming kernels: 128-bit coalesced loads, warp-shuffle and
// shared-memory reductions, one atomicMax per block and group.
#include <algorithm>
#include <type_traits>

#include "quant_device.cuh"

namespace qm {
namespace {

// ---------------------------------------------------------------- absmax, whole tensor
// Rows of `c` contiguous elements (vector loads for the multiple-of-8 part, scalar loads for
// the tail).  When the rows are dense the host flattens the tensor into a single row so that
// every block gets an equal share.
template <typename T>
__global__ void __launch_bounds__(kThreads)
absmax_tensor_kernel(const T* __restrict__ x, int64_t rows, int64_t c, int64_t row_stride,
                     const FastDiv by_vec, uint32_t* __restrict__ amax) {
  pdl_prologue();
  const int64_t vec_per_row = c >> 3;
  const int64_t total_vec = rows * vec_per_row;
  const bool narrow = total_vec < (1ll << 32);       // by_vec divides 32-bit indices by vec_per_row
  auto row_of = [&](int64_t j) { return narrow ? (int64_t)by_vec.div((uint32_t)j) : j / vec_per_row; };
  uint32_t acc = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (rows == 1) {
    // dense tensor walked as one row: no index arithmetic beyond the stride;
    // eight independent 128-bit loads in flight per thread
    for (; i + 7 * stride < total_vec; i += 8 * stride) {
      Vec8 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = Loader<T>::load8(x + (i + u * stride) * 8);
#pragma unroll
      for (int u = 0; u < 8; ++u) acc = absmax8(v[u], acc);
    }
    if (i < total_vec) {
      // remainder (fewer than eight per thread): still issued together, not one after another;
      // lanes past the end re-read the last vector, which cannot change a maximum
      Vec8 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int64_t j = i + u * stride;
        v[u] = Loader<T>::load8(x + (j < total_vec ? j : total_vec - 1) * 8);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) acc = absmax8(v[u], acc);
    }
  } else {
    // four independent 128-bit loads in flight per thread
    for (; i + 3 * stride < total_vec; i += 4 * stride) {
      Vec8 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        int64_t j = i + u * stride;
        const int64_t r = row_of(j), k = j - r * vec_per_row;
        v[u] = Loader<T>::load8(x + r * row_stride + k * 8);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) acc = absmax8(v[u], acc);
    }
    for (; i < total_vec; i += stride) {
      const int64_t r = row_of(i), k = i - r * vec_per_row;
      acc = absmax8(Loader<T>::load8(x + r * row_stride + k * 8), acc);
    }
  }
  const int64_t tail = c & 7;
  if (tail) {
    const int64_t total_tail = rows * tail;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < total_tail; j += stride) {
      int64_t r = j / tail, k = j - r * tail;
      acc = max(acc, absbits_f32(__float_as_uint(Loader<T>::load1(x, r * row_stride + (c - tail) + k))));
    }
  }
  acc = block_max(acc);
  if (threadIdx.x == 0 && acc) atomicMax(amax, acc);
}

// ---------------------------------------------------------------- absmax, dense tensor
// One flat run of 32-byte vectors (base 32-byte aligned): 256-bit loads, IN_FLIGHT of them
// outstanding per thread, and the maximum taken on packed words: for bf16 two sign-cleared 16-bit
// patterns per word (unsigned 16-bit maxima order like the magnitudes), for fp32 one 31-bit pattern.
template <typename T, int IN_FLIGHT, bool STREAM>
__global__ void __launch_bounds__(kThreads)
absmax_dense_kernel(const uint8_t* __restrict__ x, uint64_t n_vec, uint32_t* __restrict__ amax) {
  pdl_prologue();
  constexpr bool kBf16 = sizeof(T) == 2;
  const uint32_t mask = kBf16 ? 0x7fff7fffu : 0x7fffffffu;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t m = 0;
  auto fold = [&](const Vec256& v) {
    if (kBf16) {
      const uint32_t a = __vmaxu2(__vmaxu2(v.lo.x & mask, v.lo.y & mask), __vmaxu2(v.lo.z & mask, v.lo.w & mask));
      const uint32_t b = __vmaxu2(__vmaxu2(v.hi.x & mask, v.hi.y & mask), __vmaxu2(v.hi.z & mask, v.hi.w & mask));
      m = __vmaxu2(m, __vmaxu2(a, b));
    } else {
      const uint32_t a = max(max(v.lo.x & mask, v.lo.y & mask), max(v.lo.z & mask, v.lo.w & mask));
      const uint32_t b = max(max(v.hi.x & mask, v.hi.y & mask), max(v.hi.z & mask, v.hi.w & mask));
      m = max(m, max(a, b));
    }
  };
  for (; i + (IN_FLIGHT - 1) * stride < n_vec; i += IN_FLIGHT * stride) {
    Vec256 v[IN_FLIGHT];
#pragma unroll
    for (int u = 0; u < IN_FLIGHT; ++u) v[u] = ld256<STREAM>(x + (i + u * stride) * 32);
#pragma unroll
    for (int u = 0; u < IN_FLIGHT; ++u) fold(v[u]);
  }
  for (; i < n_vec; i += stride) fold(ld256<STREAM>(x + i * 32));
  uint32_t acc = kBf16 ? (max(m & 0xffffu, m >> 16) << 16) : m;      // as an fp32 bit pattern
  acc = block_max(acc);
  if (threadIdx.x == 0 && acc) atomicMax(amax, acc);
}

// ---------------------------------------------------------------- absmax per row (contiguous rows)
// G lanes share a row; rows are (batch, nc) pairs.
template <typename T, int G>
__global__ void __launch_bounds__(kThreads)
absmax_rows_kernel(const T* __restrict__ x, int64_t nc, int64_t c, int64_t s_nc, int64_t batch,
                   int64_t s_b, uint32_t* __restrict__ amax) {
  pdl_prologue();
  const int64_t rows = nc * batch;
  const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
  const int sub = threadIdx.x % G;
  uint32_t acc = 0;
  if (row < rows) {
    const int64_t b = row / nc, r = row - b * nc;
    const T* p = x + b * s_b + r * s_nc;
    const int64_t nvec = c >> 3;
    for (int64_t k = sub; k < nvec; k += G) acc = absmax8(Loader<T>::load8(p + k * 8), acc);
    for (int64_t k = (nvec << 3) + sub; k < c; k += G)
      acc = max(acc, absbits_f32(__float_as_uint(Loader<T>::load1(p, k))));
  }
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) acc = max(acc, __shfl_xor_sync(0xffffffffu, acc, o, G));
  if (row < rows && sub == 0) amax[row] = acc;
}

// ---------------------------------------------------------------- absmax per column (strided contraction)
// Storage is [c][nc] with nc contiguous; one value per column.  Each thread owns 8 adjacent
// columns; blockDim = (32, 8): 256 columns wide, 8 row slices; grid.y splits the rows.
template <typename T>
__global__ void __launch_bounds__(kThreads)
absmax_cols_kernel(const T* __restrict__ x, int64_t nc, int64_t c, int64_t s_c, int64_t s_b,
                   int64_t rows_per_block, uint32_t* __restrict__ amax) {
  pdl_prologue();
  __shared__ uint32_t s[8][256];
  const int64_t b = blockIdx.z;
  const int64_t col0 = ((int64_t)blockIdx.x * 32 + threadIdx.x) * 8;
  const int64_t r0 = (int64_t)blockIdx.y * rows_per_block;
  const int64_t r1 = min(c, r0 + rows_per_block);
  uint32_t acc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0;
  const T* base = x + b * s_b;
  if (col0 + 8 <= nc) {
    for (int64_t r = r0 + threadIdx.y; r < r1; r += 8) {
      Vec8 v = Loader<T>::load8(base + r * s_c + col0);
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i] = max(acc[i], absbits_f32(__float_as_uint(v.v[i])));
    }
  } else if (col0 < nc) {
    for (int64_t r = r0 + threadIdx.y; r < r1; r += 8)
      for (int i = 0; i < 8 && col0 + i < nc; ++i)
        acc[i] = max(acc[i], absbits_f32(__float_as_uint(Loader<T>::load1(base, r * s_c + col0 + i))));
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) s[threadIdx.y][threadIdx.x * 8 + i] = acc[i];
  __syncthreads();
  const int t = threadIdx.y * 32 + threadIdx.x;      // 0..255: one column each
  uint32_t m = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) m = max(m, s[j][t]);
  const int64_t col = (int64_t)blockIdx.x * 256 + t;
  if (col < nc && m) atomicMax(amax + b * nc + col, m);
}

// Per-channel maxima shared along the batch: batch element b belongs to group b % groups, and
// every (group, channel) entry becomes the maximum over the group's batch elements (integer max
// of the order-preserving bit patterns), written back to each of them.  One thread per entry.
__global__ void share_amax_kernel(uint32_t* __restrict__ amax, int64_t batch, int64_t groups, int64_t nc) {
  pdl_prologue();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= groups * nc) return;
  const int64_t g = i / nc, ch = i - g * nc;
  uint32_t m = 0;
  for (int64_t b = g; b < batch; b += groups) m = max(m, amax[b * nc + ch]);
  for (int64_t b = g; b < batch; b += groups) amax[b * nc + ch] = m;
}

__global__ void finalize_delta_kernel(float* __restrict__ delta, int64_t n, float qmax,
                                      uint32_t* __restrict__ err_word) {
  pdl_prologue();
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t bits = __float_as_uint(delta[i]);
  float amax = __uint_as_float(bits);
  if (bits >= 0x7f800000u && err_word) atomicOr(err_word, QM_DEVERR_NONFINITE);
  delta[i] = bits == 0 ? 1.0f : __fdiv_rn(amax, qmax);
}

// Where a quantize kernel gets its scales from.  Either finished deltas, or (from_amax) the bit
// patterns of max|x| left by an absmax kernel: the division of Eq. 1 is then done here, which
// saves a launch; the thread named `writer` stores the delta for later consumers and raises
// the non-finite flag.
struct DeltaSrc {
  const float* p;
  int per_channel;
  int from_amax;
  float qmax;
  float* out;           // from_amax only: where the finished deltas go
  uint32_t* err_word;   // from_amax only, optional
  __device__ __forceinline__ float get(int64_t i, bool writer) const {
    if (!from_amax) return __ldg(p + i);
    const uint32_t bits = __ldg(reinterpret_cast<const uint32_t*>(p) + i);
    const float d = bits == 0 ? 1.0f : __fdiv_rn(__uint_as_float(bits), qmax);
    if (writer) {
      out[i] = d;
      if (bits >= 0x7f800000u && err_word) atomicOr(err_word, QM_DEVERR_NONFINITE);
    }
    return d;
  }
};

// ---------------------------------------------------------------- quantize, contiguous contraction
// One thread handles 16 consecutive elements of a row: two 128-bit loads (bf16), one 128-bit
// code store, optionally two 128-bit stores of |x| as bf16.
template <typename T, int FMT>
__global__ void __launch_bounds__(kThreads)
quantize_rows_kernel(const T* __restrict__ x, int64_t nc, int64_t c, int64_t s_nc, int64_t batch,
                     int64_t s_b, const DeltaSrc ds, const FastDiv by_chunks, const FastDiv by_nc,
                     uint8_t* __restrict__ codes, int64_t ldc, __nv_bfloat16* __restrict__ abs_copy,
                     const Rounding rnd) {
  pdl_prologue();
  const uint32_t chunks_per_row = (uint32_t)(ldc >> 4);     // 16 codes per chunk, padding included
  const uint32_t total = (uint32_t)(nc * batch) * chunks_per_row;   // < 2^32, checked by the host
  const uint32_t stride = gridDim.x * blockDim.x;
  const float d_tensor = ds.per_channel ? 0.f : ds.get(0, blockIdx.x == 0 && threadIdx.x == 0);
  const Quotient quot_tensor(d_tensor);
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride) {
    const uint32_t row = by_chunks.div(i), ch = i - row * chunks_per_row;
    const uint32_t b = by_nc.div(row), r = row - b * (uint32_t)nc;
    const T* p = x + (int64_t)b * s_b + (int64_t)r * s_nc + ch * 16;
    const Quotient quot = ds.per_channel ? Quotient(ds.get(row, ch == 0)) : quot_tensor;
    const int64_t k0 = ch * 16;
    Vec8 v0, v1;
    if (k0 + 16 <= c) {
      v0 = Loader<T>::load8(p);
      v1 = Loader<T>::load8(p + 8);
    } else {                                                // ragged end of the row: zero fill
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        v0.v[j] = k0 + j < c ? Loader<T>::load1(p, j) : 0.f;
        v1.v[j] = k0 + 8 + j < c ? Loader<T>::load1(p, 8 + j) : 0.f;
      }
    }
    uint2 q0, q1;
    if (rnd.stochastic) {
      const uint64_t e0 = (uint64_t)row * (uint64_t)c + (uint64_t)k0;   // number of the chunk's first element
      q0 = quant8_sr<FMT>(v0, quot, rnd, e0);
      q1 = quant8_sr<FMT>(v1, quot, rnd, e0 + 8);
    } else {
      q0 = quant8<FMT>(v0, quot);
      q1 = quant8<FMT>(v1, quot);
    }
    *reinterpret_cast<uint4*>(codes + row * ldc + k0) = make_uint4(q0.x, q0.y, q1.x, q1.y);
    if (abs_copy) {
      __nv_bfloat16* a = abs_copy + row * c + k0;
      if (k0 + 16 <= c && (c & 7) == 0) {
        *reinterpret_cast<uint4*>(a) = abs_bf16x8(v0);
        *reinterpret_cast<uint4*>(a + 8) = abs_bf16x8(v1);
      } else {
        for (int j = 0; j < 8; ++j) {
          if (k0 + j < c) a[j] = __float2bfloat16_rn(fabsf(v0.v[j]));
          if (k0 + 8 + j < c) a[8 + j] = __float2bfloat16_rn(fabsf(v1.v[j]));
        }
      }
    }
  }
}

// ---------------------------------------------------------------- quantize, dense bf16 fast path
// The common case of the probe: a dense bf16 tensor whose rows are a multiple of 16 long, so the
// whole tensor is one flat run of 16-element chunks and codes have no padding.  Each thread
// takes CHUNKS chunks a block-width apart and issues all of their 128-bit loads before touching
// any of them (2 x CHUNKS loads in flight per thread; 4 for tensors that fill the GPU several
// times over, 1 for small ones, which need the parallelism more); |x| copies are the raw
// bit patterns with the sign bits cleared.
// WIDE: the tensor starts on a 32-byte boundary and a chunk is fetched with one 256-bit load (the
// four-chunk variant, used for tensors far larger than L2, also asks for evict-first).
template <int FMT, int CHUNKS, bool WIDE>
__global__ void __launch_bounds__(kThreads)
quantize_dense_kernel(const uint4* __restrict__ x, uint32_t total_chunks, const DeltaSrc ds,
                      const FastDiv by_chunks, uint32_t chunks_per_row, uint4* __restrict__ codes,
                      uint4* __restrict__ abs_copy) {
  pdl_prologue();
  const uint32_t base = blockIdx.x * (kThreads * CHUNKS) + threadIdx.x;
  uint4 w[CHUNKS][2];
#pragma unroll
  for (int u = 0; u < CHUNKS; ++u) {
    const uint32_t i = base + u * kThreads;
    const uint32_t j = i < total_chunks ? i : total_chunks - 1;     // clamp: results of dead lanes are dropped
    if (WIDE) {
      const Vec256 v = ld256<CHUNKS == 4>(x + 2 * (size_t)j);
      w[u][0] = v.lo; w[u][1] = v.hi;
    } else {
      w[u][0] = __ldg(x + 2 * (size_t)j);
      w[u][1] = __ldg(x + 2 * (size_t)j + 1);
    }
  }
  const float d_tensor = ds.per_channel ? 0.f : ds.get(0, blockIdx.x == 0 && threadIdx.x == 0);
  if (!ds.per_channel && !abs_copy && QuotientPair::serves(d_tensor)) {
    // one scale for the whole tensor: the two-wide exact quotient (guarded against overflow
    // when the scale was handed in rather than taken from the tensor's own max|x|)
    const QuotientPair qp(d_tensor);
#pragma unroll
    for (int u = 0; u < CHUNKS; ++u) {
      const uint32_t i = base + u * kThreads;
      if (i < total_chunks)
        codes[i] = ds.from_amax ? quant_bf16x16<FMT, false>(w[u][0], w[u][1], qp) : quant_bf16x16<FMT, true>(w[u][0], w[u][1], qp);
    }
    return;
  }
  const Quotient quot_tensor(d_tensor);
#pragma unroll
  for (int u = 0; u < CHUNKS; ++u) {
    const uint32_t i = base + u * kThreads;
    if (i >= total_chunks) break;
    Quotient quot = quot_tensor;
    if (ds.per_channel) {
      const uint32_t row = by_chunks.div(i);
      quot = Quotient(ds.get(row, i == row * chunks_per_row));
    }
    uint4 out;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint4 v = w[u][h];
      Vec8 f;
      f.v[0] = bf16_lo(v.x); f.v[1] = bf16_hi(v.x); f.v[2] = bf16_lo(v.y); f.v[3] = bf16_hi(v.y);
      f.v[4] = bf16_lo(v.z); f.v[5] = bf16_hi(v.z); f.v[6] = bf16_lo(v.w); f.v[7] = bf16_hi(v.w);
      const uint2 q = quant8<FMT>(f, quot);
      if (h == 0) { out.x = q.x; out.y = q.y; } else { out.z = q.x; out.w = q.y; }
      if (abs_copy) {
        const uint32_t m = 0x7fff7fffu;
        abs_copy[2 * (size_t)i + h] = make_uint4(v.x & m, v.y & m, v.z & m, v.w & m);
      }
    }
    codes[i] = out;
  }
}

// The same tensors with stochastic rounding: a thread takes one chunk of sixteen elements, four counter blocks.
// Bound by the draws (ten rounds of two wide multiplications per four elements) beside HBM: 16384 x 4096
// with its max|x| pass 138 us one element at a time, 103 us so.
template <int FMT>
__global__ void __launch_bounds__(kThreads, 4)
quantize_dense_sr_kernel(const uint4* __restrict__ x, uint32_t total_chunks, const DeltaSrc ds, const FastDiv by_chunks,
                         uint32_t chunks_per_row, uint4* __restrict__ codes, const Rounding rnd) {
  pdl_prologue();
  const uint32_t i = blockIdx.x * kThreads + threadIdx.x;
  if (i >= total_chunks) return;
  const uint4 a = __ldg(x + 2 * (size_t)i), b = __ldg(x + 2 * (size_t)i + 1);
  uint32_t row = 0;
  if (ds.per_channel) row = by_chunks.div(i);
  const float d = ds.per_channel ? ds.get(row, i == row * chunks_per_row) : ds.get(0, i == 0);
  const uint64_t number = (uint64_t)i * 16u;              // of the chunk's first element: rows are dense
  if (QuotientPair::serves(d)) {
    const QuotientPair qp(d);
    codes[i] = ds.from_amax ? quant_bf16x16_sr<FMT, false>(a, b, qp, rnd, number) : quant_bf16x16_sr<FMT, true>(a, b, qp, rnd, number);
    return;
  }
  const Quotient quot(d);
  const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  Vec8 f[2];
#pragma unroll
  for (int h = 0; h < 8; ++h) { f[h >> 2].v[2 * (h & 3)] = bf16_lo(w[h]); f[h >> 2].v[2 * (h & 3) + 1] = bf16_hi(w[h]); }
  const uint2 q0 = quant8_sr<FMT, true>(f[0], quot, rnd, number), q1 = quant8_sr<FMT, true>(f[1], quot, rnd, number + 8);
  codes[i] = make_uint4(q0.x, q0.y, q1.x, q1.y);
}

// ---------------------------------------------------------------- several formats in one pass
// A sweep of formats quantizes the same tensor two or three times (Table 1).  These kernels read
// it once and write the codes of every format in MASK (bit f = qm_format f), with per-tensor
// scales taken from the tensor's max|x| bit pattern: delta_f = max|x| / qmax_f.  Thread 0 of
// block 0 stores the scales and raises the non-finite flag for each format's probe.
struct MultiOut {
  uint8_t* codes[3];      // indexed by qm_format; null where MASK has no bit
  float* delta_out[3];
  uint32_t* err_word[3];
};

template <int MASK>
__device__ __forceinline__ void multi_scales(const uint32_t* amax, const MultiOut& o, bool writer, float (&d)[3]) {
  const uint32_t bits = __ldg(amax);
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    if (!(MASK & (1 << f))) { d[f] = 1.f; continue; }
    d[f] = bits == 0 ? 1.0f : __fdiv_rn(__uint_as_float(bits), fmt_qmax(f));
    if (writer) {
      o.delta_out[f][0] = d[f];
      if (bits >= 0x7f800000u && o.err_word[f]) atomicOr(o.err_word[f], QM_DEVERR_NONFINITE);
    }
  }
}

// ---------------------------------------------------------------- sixteen elements as they come
template <typename T> struct Piece;
template <> struct Piece<__nv_bfloat16> {
  uint4 w[2];
  __device__ __forceinline__ void load(const __nv_bfloat16* p, bool wide) {
    if (wide) { const Vec256 v = ld256<false>(p); w[0] = v.lo; w[1] = v.hi; }
    else { w[0] = __ldg(reinterpret_cast<const uint4*>(p)); w[1] = __ldg(reinterpret_cast<const uint4*>(p) + 1); }
  }
  __device__ __forceinline__ void zero() { w[0] = w[1] = make_uint4(0u, 0u, 0u, 0u); }
  // the n < 16 elements that are left of a line, zeros behind them
  __device__ __forceinline__ void load_part(const __nv_bfloat16* p, int n) {
    const bool half = n >= 8;
    const unsigned short* e = reinterpret_cast<const unsigned short*>(p) + (half ? 8 : 0);
    const int m = half ? n - 8 : n;
    uint32_t h[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) h[j] = j < m ? (uint32_t)__ldg(e + j) : 0u;
    const uint4 v = make_uint4(h[0] | h[1] << 16, h[2] | h[3] << 16, h[4] | h[5] << 16, h[6] | h[7] << 16), z = make_uint4(0u, 0u, 0u, 0u);
    w[0] = half ? __ldg(reinterpret_cast<const uint4*>(p)) : v;
    w[1] = half ? v : z;
  }
  __device__ __forceinline__ uint32_t absmax() const {    // as an fp32 bit pattern
    const uint32_t k = 0x7fff7fffu;
    uint32_t m = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h)
      m = __vmaxu2(m, __vmaxu2(__vmaxu2(w[h].x & k, w[h].y & k), __vmaxu2(w[h].z & k, w[h].w & k)));
    return max(m & 0xffffu, m >> 16) << 16;
  }
  template <int FMT, bool GUARD = false> __device__ __forceinline__ uint4 quant(const QuotientPair& qp) const { return quant_bf16x16<FMT, GUARD>(w[0], w[1], qp); }
  __device__ __forceinline__ float at(int i) const {
    const uint4 v = w[i >> 3];
    const uint32_t x = (i >> 1 & 3) == 0 ? v.x : (i >> 1 & 3) == 1 ? v.y : (i >> 1 & 3) == 2 ? v.z : v.w;
    return i & 1 ? bf16_hi(x) : bf16_lo(x);
  }
};
template <> struct Piece<float> {
  float4 w[4];
  __device__ __forceinline__ void load(const float* p, bool) {
#pragma unroll
    for (int h = 0; h < 4; ++h) w[h] = __ldg(reinterpret_cast<const float4*>(p) + h);
  }
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int h = 0; h < 4; ++h) w[h] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __device__ __forceinline__ void load_part(const float* p, int n) {
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      if (4 * h + 4 <= n) { w[h] = __ldg(reinterpret_cast<const float4*>(p) + h); continue; }
      float e[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) e[j] = 4 * h + j < n ? __ldg(p + 4 * h + j) : 0.f;
      w[h] = make_float4(e[0], e[1], e[2], e[3]);
    }
  }
  __device__ __forceinline__ uint32_t absmax() const {
    uint32_t m = 0;
#pragma unroll
    for (int h = 0; h < 4; ++h)
      m = max(m, max(max(absbits_f32(__float_as_uint(w[h].x)), absbits_f32(__float_as_uint(w[h].y))),
                     max(absbits_f32(__float_as_uint(w[h].z)), absbits_f32(__float_as_uint(w[h].w)))));
    return m;
  }
  template <int FMT, bool GUARD = false> __device__ __forceinline__ uint4 quant(const QuotientPair& qp) const {
    uint32_t c[4];
#pragma unroll
    for (int h = 0; h < 4; ++h)
      c[h] = quant_pair_x2<FMT, GUARD>(w[h].x, w[h].y, qp) | quant_pair_x2<FMT, GUARD>(w[h].z, w[h].w, qp) << 16;
    return make_uint4(c[0], c[1], c[2], c[3]);
  }
  __device__ __forceinline__ float at(int i) const {
    const float4 v = w[i >> 2];
    return (i & 3) == 0 ? v.x : (i & 3) == 1 ? v.y : (i & 3) == 2 ? v.z : v.w;
  }
};

// ---------------------------------------------------------------- quantize, lines of any length and pitch under one scale
// What the dense kernels do not take: bf16 rows that are no multiple of 16 long or lie apart, and fp32.  A thread takes
// sixteen elements of a line, every format in MASK, with the two-wide quotient; of a line's last piece only the loads are
// element by element (with its arithmetic so too, every warp that held one took 1.3 to 1.8 x as long).  Bound by HBM; us per
// call, one element at a time and a launch per format / last piece one at a time / so: 13809 x 1234 bf16 under a given scale
// 14.9 / 13.6 / 12.1, three formats with their max|x| pass 61.6 / 51.3 / 31.9; fp32 16384 x 4096 57 / 49 and 222 / 121.
// 128 x 40 x 128 in a batch of 512, the right operand strided, three formats: transposed 72.4, 78.4, so 71.1.
template <typename T, int MASK, bool GUARD>
__global__ void __launch_bounds__(kThreads)
quantize_lines_kernel(const T* __restrict__ x, uint32_t total, int64_t c, int64_t s_nc, int64_t s_b, const FastDiv by_chunks,
                      const FastDiv by_nc, const uint32_t* __restrict__ amax, const float* __restrict__ delta, const MultiOut o,
                      int64_t ldc) {
  pdl_prologue();
  const uint32_t i = blockIdx.x * kThreads + threadIdx.x;
  if (i >= total) return;
  const uint32_t row = by_chunks.div(i), ch = i - row * by_chunks.d, b = by_nc.div(row);
  const int64_t k0 = (int64_t)ch * 16;
  const T* src = x + (int64_t)b * s_b + (int64_t)(row - b * by_nc.d) * s_nc + k0;
  const bool whole = k0 + 16 <= c;
  Piece<T> p;
  if (whole) p.load(src, false); else p.load_part(src, (int)(c - k0));
  float d[3] = {1.f, 1.f, 1.f};
  if (GUARD) {
    const float given = __ldg(delta);
#pragma unroll
    for (int f = 0; f < 3; ++f) d[f] = given;
  } else {
    multi_scales<MASK>(amax, o, i == 0, d);
  }
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    if (!(MASK & (1 << f))) continue;
    uint4* dst = reinterpret_cast<uint4*>(o.codes[f] + (int64_t)row * ldc + k0);
    if (QuotientPair::serves(d[f])) {
      const QuotientPair qp(d[f]);
      *dst = f == 0 ? p.template quant<0, GUARD>(qp) : f == 1 ? p.template quant<1, GUARD>(qp) : p.template quant<2, GUARD>(qp);
    } else {
      const Quotient quot(d[f]);
      uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int e = 0; e < 16; e += 2) {
        const float t0 = quot(p.at(e)), t1 = quot(p.at(e + 1));
        w[e >> 2] |= (f == 0 ? quant2<0>(t0, t1) : f == 1 ? quant2<1>(t0, t1) : quant2<2>(t0, t1)) << (16 * (e >> 1 & 1));
      }
      *dst = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

// Dense bf16 tensor, rows a multiple of 16 long: one flat run of 16-element chunks.
template <int MASK, int CHUNKS, bool WIDE>
__global__ void __launch_bounds__(kThreads)
quantize_dense_multi_kernel(const uint4* __restrict__ x, uint32_t total_chunks, const uint32_t* __restrict__ amax,
                            const MultiOut o) {
  pdl_prologue();
  const uint32_t base = blockIdx.x * (kThreads * CHUNKS) + threadIdx.x;
  uint4 w[CHUNKS][2];
#pragma unroll
  for (int u = 0; u < CHUNKS; ++u) {
    const uint32_t i = base + u * kThreads;
    const uint32_t j = i < total_chunks ? i : total_chunks - 1;     // clamp: results of dead lanes are dropped
    if (WIDE) {
      const Vec256 v = ld256<CHUNKS == 4>(x + 2 * (size_t)j);
      w[u][0] = v.lo; w[u][1] = v.hi;
    } else {
      w[u][0] = __ldg(x + 2 * (size_t)j);
      w[u][1] = __ldg(x + 2 * (size_t)j + 1);
    }
  }
  float d[3];
  multi_scales<MASK>(amax, o, blockIdx.x == 0 && threadIdx.x == 0, d);
  const bool pair_ok = QuotientPair::serves(d[0]) && QuotientPair::serves(d[1]) && QuotientPair::serves(d[2]);
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    if (!(MASK & (1 << f))) continue;
    uint4* codes = reinterpret_cast<uint4*>(o.codes[f]);
    if (pair_ok) {
      const QuotientPair quot(d[f]);
#pragma unroll
      for (int u = 0; u < CHUNKS; ++u) {
        const uint32_t i = base + u * kThreads;
        if (i < total_chunks) {
          codes[i] = f == 0   ? quant_bf16x16<0>(w[u][0], w[u][1], quot)
                     : f == 1 ? quant_bf16x16<1>(w[u][0], w[u][1], quot)
                              : quant_bf16x16<2>(w[u][0], w[u][1], quot);
        }
      }
    } else {
      const Quotient quot(d[f]);
#pragma unroll 1
      for (int u = 0; u < CHUNKS; ++u) {
        const uint32_t i = base + u * kThreads;
        if (i >= total_chunks) break;
        uint4 out;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint4 v = w[u][h];
          Vec8 t;
          t.v[0] = bf16_lo(v.x); t.v[1] = bf16_hi(v.x); t.v[2] = bf16_lo(v.y); t.v[3] = bf16_hi(v.y);
          t.v[4] = bf16_lo(v.z); t.v[5] = bf16_hi(v.z); t.v[6] = bf16_lo(v.w); t.v[7] = bf16_hi(v.w);
          const uint2 q = f == 0 ? quant8<0>(t, quot) : f == 1 ? quant8<1>(t, quot) : quant8<2>(t, quot);
          if (h == 0) { out.x = q.x; out.y = q.y; } else { out.z = q.x; out.w = q.y; }
        }
        codes[i] = out;
      }
    }
  }
}

// ---------------------------------------------------------------- quantize + transpose through shared memory
// Storage [c][nc] (nc contiguous, bf16), c a multiple of 16 (EDGE: c not a multiple of 128 or nc not one of 64;
// rows and columns beyond the matrix are loaded as zeros and not written).  A block
// takes a tile of 128 contraction rows x 64 columns: it loads the tile with whole-line reads (8
// threads per 128-byte row), reads it back column-wise (a thread takes 16 contraction entries of two
// adjacent columns; consecutive lanes read consecutive words: conflict-free), quantizes, and hands
// the codes (128 bytes per output row and format) and the contraction-major copy (256 bytes per
// output row) to global memory through a second shared-memory tile so that every store instruction
// writes whole lines: 16-byte chunk ch of output row n sits at ch ^ ((n >> 1) & 7), which keeps
// both the column-wise writes and the row-wise reads of that tile conflict-free.
template <int MASK> struct TileSmem {
  static constexpr int kFormats = (MASK & 1) + (MASK >> 1 & 1) + (MASK >> 2 & 1);
  static constexpr int kVec = kFormats * 64 * 8 + 64 * 16;        // 16-byte units: 24, 32 or 40 KB for one, two or three formats
  static __device__ __forceinline__ int slot(int f) { return (f > 0 ? MASK & 1 : 0) + (f > 1 ? MASK >> 1 & 1 : 0); }
};
// d_lo / d_hi: the scales of the thread's two columns, per format in MASK (bit f = qm_format f).
// tile: column tile, contraction tile, batch element.  SR: stochastic rounding (rnd); c is a multiple of 4, so sixteen entries are four counter blocks.
template <int MASK, bool GUARD, bool EDGE, bool SR = false>
__device__ __forceinline__ void transpose_tile(const __nv_bfloat16* __restrict__ x, int64_t nc, int64_t c, int64_t s_c,
                                               int64_t s_b, const float (&d_lo)[3], const float (&d_hi)[3],
                                               uint8_t* const (&codes)[3], int64_t ldc,
                                               __nv_bfloat16* __restrict__ kmaj_copy, uint4* smem, const uint3 tile,
                                               const Rounding& rnd = Rounding{}) {
  const int t = threadIdx.x;
  const int64_t b = tile.z, n0 = (int64_t)tile.x * 64, k0 = (int64_t)tile.y * 128;
  const int64_t pitch = s_c >> 3;                                     // row stride in 16-byte units
  // 128 rows x 128 bytes, four 16-byte loads per thread in flight
  auto fetch = [&](uint4 (&v)[4]) {
    const uint4* src = reinterpret_cast<const uint4*>(x + b * s_b + k0 * s_c + n0);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t at = (int64_t)((t >> 3) + 32 * i) * pitch + (t & 7);
      if (!EDGE) {
        v[i] = __ldg(src + at);
      } else {
        const int64_t left = nc - (n0 + 8 * (t & 7));                // columns of this vector that exist
        v[i] = make_uint4(0u, 0u, 0u, 0u);
        if (k0 + (t >> 3) + 32 * i < c && left > 0) {
          if (left >= 8) {
            v[i] = __ldg(src + at);
          } else {
            const unsigned short* e = reinterpret_cast<const unsigned short*>(src + at);
            uint32_t h[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) h[j] = j < left ? (uint32_t)__ldg(e + j) : 0u;
            v[i] = make_uint4(h[0] | h[1] << 16, h[2] | h[3] << 16, h[4] | h[5] << 16, h[6] | h[7] << 16);
          }
        }
      }
    }
  };
  // phase 1: the tile into shared memory
  {
    uint4 v[4];
    fetch(v);
#pragma unroll
    for (int i = 0; i < 4; ++i) smem[((t >> 3) + 32 * i) * 8 + (t & 7)] = v[i];
  }
  __syncthreads();
  // phase 2: columns 2p, 2p + 1, contraction entries 16g .. 16g + 15
  const int pcol = t & 31, g = t >> 5;
  uint32_t w[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) w[j] = reinterpret_cast<const uint32_t*>(smem)[(16 * g + j) * 32 + pcol];
  __syncthreads();                                                     // the output tiles reuse the input tile's memory
  uint4* const s_codes = smem;                                         // [formats][64 rows][8 chunks]
  uint4* const s_kmaj = s_codes + TileSmem<MASK>::kFormats * 64 * 8;   // [64 rows][16 chunks]
  const uint32_t sw = (uint32_t)pcol & 7u;
#pragma unroll SR ? 1 : 2
  for (int col = 0; col < 2; ++col) {
    const int n = 2 * pcol + col;
    uint32_t pw[8];                                                    // this column's 16 values, two bf16 per word
#pragma unroll
    for (int j = 0; j < 8; ++j)
      pw[j] = __byte_perm(w[2 * j], w[2 * j + 1], col == 0 ? 0x5410 : 0x7632);
    const uint4 a = make_uint4(pw[0], pw[1], pw[2], pw[3]), bb = make_uint4(pw[4], pw[5], pw[6], pw[7]);
    if (kmaj_copy) {
      s_kmaj[n * 16 + ((2 * g) ^ sw)] = a;
      s_kmaj[n * 16 + ((2 * g + 1) ^ sw)] = bb;
    }
    // what lies beyond the matrix is not written; its zeros would take the slow branch of stochastic rounding
    if (EDGE && (n0 + n >= nc || k0 + 16 * g >= c)) continue;
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      if (!(MASK & (1 << f))) continue;
      const float d = col == 0 ? d_lo[f] : d_hi[f];
      uint4 cw;
      const uint64_t number = (uint64_t)(b * nc + n0 + n) * (uint64_t)c + (uint64_t)(k0 + 16 * g);    // of the first entry
      if (QuotientPair::serves(d)) {
        const QuotientPair qp(d);
        if (SR) cw = f == 0 ? quant_bf16x16_sr<0, GUARD>(a, bb, qp, rnd, number) : f == 1 ? quant_bf16x16_sr<1, GUARD>(a, bb, qp, rnd, number) : quant_bf16x16_sr<2, GUARD>(a, bb, qp, rnd, number);
        else cw = f == 0 ? quant_bf16x16<0, GUARD>(a, bb, qp) : f == 1 ? quant_bf16x16<1, GUARD>(a, bb, qp) : quant_bf16x16<2, GUARD>(a, bb, qp);
      } else {
        const Quotient quot(d);
        Vec8 lo, hi;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          lo.v[2 * j] = bf16_lo(pw[j]); lo.v[2 * j + 1] = bf16_hi(pw[j]);
          hi.v[2 * j] = bf16_lo(pw[4 + j]); hi.v[2 * j + 1] = bf16_hi(pw[4 + j]);
        }
        uint2 q0, q1;
        if (SR) {
          q0 = f == 0 ? quant8_sr<0, true>(lo, quot, rnd, number) : f == 1 ? quant8_sr<1, true>(lo, quot, rnd, number) : quant8_sr<2, true>(lo, quot, rnd, number);
          q1 = f == 0 ? quant8_sr<0, true>(hi, quot, rnd, number + 8) : f == 1 ? quant8_sr<1, true>(hi, quot, rnd, number + 8) : quant8_sr<2, true>(hi, quot, rnd, number + 8);
        } else {
          q0 = f == 0 ? quant8<0>(lo, quot) : f == 1 ? quant8<1>(lo, quot) : quant8<2>(lo, quot);
          q1 = f == 0 ? quant8<0>(hi, quot) : f == 1 ? quant8<1>(hi, quot) : quant8<2>(hi, quot);
        }
        cw = make_uint4(q0.x, q0.y, q1.x, q1.y);
      }
      s_codes[(TileSmem<MASK>::slot(f) * 64 + n) * 8 + ((uint32_t)g ^ sw)] = cw;
    }
  }
  __syncthreads();
  // phase 3: whole output rows
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    if (!(MASK & (1 << f))) continue;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int row = (t >> 3) + 32 * i, ch = t & 7;
      if (EDGE && (n0 + row >= nc || k0 + ch * 16 >= ldc)) continue;
      const uint4 v = s_codes[(TileSmem<MASK>::slot(f) * 64 + row) * 8 + (ch ^ ((row >> 1) & 7))];
      *reinterpret_cast<uint4*>(codes[f] + (b * nc + n0 + row) * ldc + k0 + ch * 16) = v;
    }
  }
  if (kmaj_copy) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int row = (t >> 4) + 16 * i, ch = t & 15;
      if (EDGE && (n0 + row >= nc || k0 + ch * 8 >= c)) continue;
      const uint4 v = s_kmaj[row * 16 + (ch ^ ((row >> 1) & 7))];
      *reinterpret_cast<uint4*>(kmaj_copy + (b * nc + n0 + row) * c + k0 + ch * 8) = v;
    }
  }
}

// One format, scales from a DeltaSrc (per tensor or per output row, finished or from max|x|).
template <int FMT, bool EDGE, bool SR>
__device__ __forceinline__ void quantize_transpose_tile(const __nv_bfloat16* __restrict__ x, int64_t nc, int64_t c, int64_t s_c,
                                                        int64_t s_b, const DeltaSrc& ds, uint8_t* __restrict__ codes, int64_t ldc,
                                                        __nv_bfloat16* __restrict__ kmaj_copy, const Rounding& rnd, uint4* smem) {
  const int pcol = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int64_t col = (int64_t)blockIdx.x * 64 + 2 * pcol, orow = (int64_t)blockIdx.z * nc + col;
  float d_lo[3] = {1.f, 1.f, 1.f}, d_hi[3] = {1.f, 1.f, 1.f};
  if (ds.per_channel) {
    if (!EDGE || col < nc) d_lo[FMT] = ds.get(orow, blockIdx.y == 0 && g == 0);
    if (!EDGE || col + 1 < nc) d_hi[FMT] = ds.get(orow + 1, blockIdx.y == 0 && g == 0);
  } else {
    d_lo[FMT] = d_hi[FMT] = ds.get(0, blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0);
  }
  uint8_t* const cd[3] = {codes, codes, codes};
  if (ds.from_amax) transpose_tile<1 << FMT, false, EDGE, SR>(x, nc, c, s_c, s_b, d_lo, d_hi, cd, ldc, kmaj_copy, smem, blockIdx, rnd);
  else transpose_tile<1 << FMT, true, EDGE, SR>(x, nc, c, s_c, s_b, d_lo, d_hi, cd, ldc, kmaj_copy, smem, blockIdx, rnd);
}

// Bound by HBM and by how many blocks hide the tile's load, compute and store phases: no second launch bound, with
// one (even of 1) the compiler takes 69 to 77 registers instead of 48 to 52, three blocks on an SM instead of
// four (INT8 codes of 16384 x 4096 under given scales: 56.0 us so, 44.6 without).
template <int FMT, bool EDGE>
__global__ void __launch_bounds__(kThreads)
quantize_transpose_tile_kernel(const __nv_bfloat16* __restrict__ x, int64_t nc, int64_t c, int64_t s_c, int64_t s_b,
                               const DeltaSrc ds, uint8_t* __restrict__ codes, int64_t ldc, __nv_bfloat16* __restrict__ kmaj_copy) {
  pdl_prologue();
  __shared__ uint4 smem[TileSmem<1 << FMT>::kVec];
  quantize_transpose_tile<FMT, EDGE, false>(x, nc, c, s_c, s_b, ds, codes, ldc, kmaj_copy, Rounding{}, smem);
}
// Stochastic rounding, bound by its draws: three blocks on an SM.
template <int FMT, bool EDGE>
__global__ void __launch_bounds__(kThreads, 3)
quantize_transpose_tile_sr_kernel(const __nv_bfloat16* __restrict__ x, int64_t nc, int64_t c, int64_t s_c, int64_t s_b,
                                  const DeltaSrc ds, uint8_t* __restrict__ codes, int64_t ldc,
                                  __nv_bfloat16* __restrict__ kmaj_copy, const Rounding rnd) {
  pdl_prologue();
  __shared__ uint4 smem[TileSmem<1 << FMT>::kVec];
  quantize_transpose_tile<FMT, EDGE, true>(x, nc, c, s_c, s_b, ds, codes, ldc, kmaj_copy, rnd, smem);
}

// Every format in MASK from one read, per-tensor scales from the tensor's max|x|.
template <int MASK, bool EDGE>
__global__ void __launch_bounds__(kThreads)
quantize_transpose_tile_multi_kernel(const __nv_bfloat16* __restrict__ x, int64_t nc, int64_t c, int64_t s_c,
                                     int64_t s_b, const uint32_t* __restrict__ amax, const MultiOut o, int64_t ldc,
                                     __nv_bfloat16* __restrict__ kmaj_copy) {
  pdl_prologue();
  __shared__ uint4 smem[TileSmem<MASK>::kVec];
  float d[3];
  multi_scales<MASK>(amax, o, blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0, d);
  uint8_t* const cd[3] = {o.codes[0], o.codes[1], o.codes[2]};
  transpose_tile<MASK, false, EDGE>(x, nc, c, s_c, s_b, d, d, cd, ldc, kmaj_copy, smem, blockIdx);
}

// ---------------------------------------------------------------- fused per-row scale + quantize
// G lanes own one row: pass 1 reduces max|x| over the row, pass 2 re-reads it (from L1/L2: the
// same lanes touched it a moment ago) and writes codes.  HBM sees each element once.
template <typename T, int FMT, int G>
__device__ __forceinline__ void scale_quantize_rows(const T* __restrict__ x, int64_t nc, int64_t c, int64_t s_nc,
                                                    int64_t batch, int64_t s_b, float qmax, float* __restrict__ delta_out,
                                                    uint8_t* __restrict__ codes, int64_t ldc,
                                                    __nv_bfloat16* __restrict__ abs_copy, uint32_t* __restrict__ err_word,
                                                    int64_t block) {
  const int64_t rows = nc * batch;
  const int64_t row = (block * blockDim.x + threadIdx.x) / G;
  const int sub = threadIdx.x % G;
  const bool live = row < rows;
  const int64_t b = live ? row / nc : 0, r = live ? row - b * nc : 0;
  const T* p = x + b * s_b + r * s_nc;
  const int64_t nvec = c >> 3;
  uint32_t acc = 0;
  if (live) {
    for (int64_t k = sub; k < nvec; k += G) acc = absmax8(Loader<T>::load8(p + k * 8), acc);
    for (int64_t k = (nvec << 3) + sub; k < c; k += G)
      acc = max(acc, absbits_f32(__float_as_uint(Loader<T>::load1(p, k))));
  }
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) acc = max(acc, __shfl_xor_sync(0xffffffffu, acc, o, G));
  if (!live) return;
  const float d = acc == 0 ? 1.0f : __fdiv_rn(__uint_as_float(acc), qmax);
  if (sub == 0) {
    delta_out[row] = d;
    if (acc >= 0x7f800000u && err_word) atomicOr(err_word, QM_DEVERR_NONFINITE);
  }
  const Quotient quot(d);
  const bool pair_ok = sizeof(T) == 2 && !abs_copy && QuotientPair::serves(d);
  const QuotientPair qp(pair_ok ? d : 1.f);                 // the row's own scale: nothing can overflow
  const int64_t nchunk = ldc >> 3;                          // 8 codes per step, padding included
  for (int64_t k = sub; k < nchunk; k += G) {
    const int64_t k0 = k * 8;
    if (pair_ok && k0 + 8 <= c) {
      const uint4 raw = __ldg(reinterpret_cast<const uint4*>(p + k0));
      *reinterpret_cast<uint2*>(codes + row * ldc + k0) = quant_bf16x8<FMT>(raw, qp);
      continue;
    }
    Vec8 v;
    if (k0 + 8 <= c) v = Loader<T>::load8(p + k0);
    else {
#pragma unroll
      for (int j = 0; j < 8; ++j) v.v[j] = k0 + j < c ? Loader<T>::load1(p, k0 + j) : 0.f;
    }
    *reinterpret_cast<uint2*>(codes + row * ldc + k0) = quant8<FMT>(v, quot);
    if (abs_copy) {
      __nv_bfloat16* a = abs_copy + row * c + k0;
      if (k0 + 8 <= c && (c & 7) == 0) *reinterpret_cast<uint4*>(a) = abs_bf16x8(v);
      else
        for (int j = 0; j < 8 && k0 + j < c; ++j) a[j] = __float2bfloat16_rn(fabsf(v.v[j]));
    }
  }
}

template <typename T, int FMT, int G>
__global__ void __launch_bounds__(kThreads)
scale_quantize_rows_kernel(const T* __restrict__ x, int64_t nc, int64_t c, int64_t s_nc,
                           int64_t batch, int64_t s_b, float qmax, float* __restrict__ delta_out,
                           uint8_t* __restrict__ codes, int64_t ldc,
                           __nv_bfloat16* __restrict__ abs_copy, uint32_t* __restrict__ err_word) {
  pdl_prologue();
  scale_quantize_rows<T, FMT, G>(x, nc, c, s_nc, batch, s_b, qmax, delta_out, codes, ldc, abs_copy, err_word, blockIdx.x);
}

// ---------------------------------------------------------------- fused per-row, row held in registers
// bf16 rows of at most VPL * 256 elements (a multiple of 16): one warp per row loads the whole row
// with VPL independent 128-bit loads per lane, reduces max|x| with shuffles, and quantizes from
// the registers.  Every element crosses the memory system once.
template <int FMT, int VPL>
__global__ void __launch_bounds__(kThreads)
scale_quantize_rows_reg_kernel(const __nv_bfloat16* __restrict__ x, int64_t nc, int nvec, int64_t s_nc,
                               int64_t batch, int64_t s_b, float qmax, float* __restrict__ delta_out,
                               uint2* __restrict__ codes, uint4* __restrict__ abs_copy,
                               uint32_t* __restrict__ err_word) {
  pdl_prologue();
  const int64_t rows = nc * batch;
  const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (row >= rows) return;                                  // whole warps leave together
  const int64_t b = row / nc, r = row - b * nc;
  const uint4* p = reinterpret_cast<const uint4*>(x + b * s_b + r * s_nc);
  uint4 w[VPL];
#pragma unroll
  for (int u = 0; u < VPL; ++u) {
    const int k = lane + 32 * u;
    w[u] = k < nvec ? __ldg(p + k) : make_uint4(0u, 0u, 0u, 0u);
  }
  // max over sign-cleared 16-bit patterns, two per word
  uint32_t m2 = 0;
#pragma unroll
  for (int u = 0; u < VPL; ++u) {
    const uint32_t k = 0x7fff7fffu;
    m2 = __vmaxu2(m2, __vmaxu2(__vmaxu2(w[u].x & k, w[u].y & k), __vmaxu2(w[u].z & k, w[u].w & k)));
  }
  uint32_t acc = max(m2 & 0xffffu, m2 >> 16) << 16;         // as an fp32 bit pattern
  acc = warp_max(acc);
  const float d = acc == 0 ? 1.0f : __fdiv_rn(__uint_as_float(acc), qmax);
  if (lane == 0) {
    delta_out[row] = d;
    if (acc >= 0x7f800000u && err_word) atomicOr(err_word, QM_DEVERR_NONFINITE);
  }
  if (!abs_copy && QuotientPair::serves(d)) {
    const QuotientPair qp(d);                                // the row's own scale: nothing can overflow
#pragma unroll
    for (int u = 0; u < VPL; ++u) {
      const int k = lane + 32 * u;
      if (k < nvec) codes[row * nvec + k] = quant_bf16x8<FMT>(w[u], qp);
    }
    return;
  }
  const Quotient quot(d);
#pragma unroll
  for (int u = 0; u < VPL; ++u) {
    const int k = lane + 32 * u;
    if (k >= nvec) break;
    const uint4 v = w[u];
    Vec8 f;
    f.v[0] = bf16_lo(v.x); f.v[1] = bf16_hi(v.x); f.v[2] = bf16_lo(v.y); f.v[3] = bf16_hi(v.y);
    f.v[4] = bf16_lo(v.z); f.v[5] = bf16_hi(v.z); f.v[6] = bf16_lo(v.w); f.v[7] = bf16_hi(v.w);
    codes[row * nvec + k] = quant8<FMT>(f, quot);
    if (abs_copy) {
      const uint32_t m = 0x7fff7fffu;
      abs_copy[row * nvec + k] = make_uint4(v.x & m, v.y & m, v.z & m, v.w & m);
    }
  }
}

// ---------------------------------------------------------------- fused per-row, a row spread over a group of warps
// Rows of at most 512 W V elements (a multiple of 16), every format in MASK: W warps share a row, a thread holds V pieces of
// sixteen elements of it, fetched with whole 256-bit loads (two 128-bit ones where rows do not start on 32 bytes) while the
// row before is reduced and quantized; one 128-bit store of codes per piece and format.  Every element crosses the memory
// system once.  Bound by HBM and instruction issue: what a thread does once per row (division, reciprocal, maxima) is why a
// thread takes two pieces.  us, a warp per row that read it twice (L1) / so: 16384 x 4096 bf16 INT8 49.3 / 35.3 (one piece
// 43.7), 4096 x 8192 39.9 / 20.0, 128 x 4096 6.7 / 3.0, 16384 x 2064 28.9 / 27.0; fp32 16384 x 4096 102 / 56, x 1024 24.3 / 17.9.
// Bf16 rows of at most 1024 stay with a warp per row (768 11.4 / 12.5), fp32 rows below 272 too (256 31.8, 128 6.5 / 7.1).
template <typename T, int MASK, int W, int V>
__global__ void __launch_bounds__(kThreads)
scale_quantize_rows_spread_kernel(const T* __restrict__ x, uint32_t rows, int pieces, int64_t s_nc, int64_t s_b, const FastDiv by_nc,
                                  const MultiOut o, bool wide) {
  pdl_prologue();
  constexpr int kRowsPerBlock = 8 / W;
  __shared__ __align__(16) uint32_t s_max[2][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int group = warp / W, t = threadIdx.x - group * (32 * W);       // the row's group of warps, thread within it
  const uint32_t step = gridDim.x * kRowsPerBlock;
  auto fetch = [&](uint32_t row, Piece<T> (&p)[V]) {
    const uint32_t b = by_nc.div(row);
    const T* src = x + (int64_t)b * s_b + (int64_t)(row - b * by_nc.d) * s_nc;
#pragma unroll
    for (int u = 0; u < V; ++u) {
      const int k = t + u * 32 * W;
      if (k < pieces) p[u].load(src + (int64_t)k * 16, wide); else p[u].zero();
    }
  };
  uint32_t row = blockIdx.x * kRowsPerBlock + group;
  if (row >= rows) return;                                              // (whole groups)
  Piece<T> next[V];
  fetch(row, next);
  for (uint32_t it = 0; row < rows; ++it) {
    Piece<T> p[V];
#pragma unroll
    for (int u = 0; u < V; ++u) p[u] = next[u];
    const uint32_t row_next = row + step;
    if (row_next < rows) fetch(row_next, next);
    uint32_t m = 0;
#pragma unroll
    for (int u = 0; u < V; ++u) m = max(m, p[u].absmax());
    m = __reduce_max_sync(0xffffffffu, m);
    if (W > 1) {                                                        // two sets of slots: one barrier per row is enough
      if (lane == 0) s_max[it & 1][warp] = m;
      asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(32 * W) : "memory");
      if (W == 2) {
        const uint2 a = *reinterpret_cast<const uint2*>(&s_max[it & 1][group * W]);
        m = max(a.x, a.y);
      } else {
#pragma unroll
        for (int j = 0; j < W; j += 4) {
          const uint4 a = *reinterpret_cast<const uint4*>(&s_max[it & 1][(group * W + j) & 4]);
          m = max(max(m, max(a.x, a.y)), max(a.z, a.w));
        }
      }
    }
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      if (!(MASK & (1 << f))) continue;
      const float d = m == 0 ? 1.0f : __fdiv_rn(__uint_as_float(m), fmt_qmax(f));
      if (t == 0) {
        o.delta_out[f][row] = d;
        if (m >= 0x7f800000u && o.err_word[f]) atomicOr(o.err_word[f], QM_DEVERR_NONFINITE);
      }
      uint4* dst = reinterpret_cast<uint4*>(o.codes[f]) + (int64_t)row * pieces;
      if (QuotientPair::serves(d)) {
        const QuotientPair qp(d);                                       // the row's own scale: nothing can overflow
#pragma unroll
        for (int u = 0; u < V; ++u) {
          const int k = t + u * 32 * W;
          if (k < pieces) dst[k] = f == 0 ? p[u].template quant<0>(qp) : f == 1 ? p[u].template quant<1>(qp) : p[u].template quant<2>(qp);
        }
      } else {
        const Quotient quot(d);
#pragma unroll 1
        for (int k = t, u = 0; k < pieces; k += 32 * W, ++u) {          // rare: scales outside 2^-60 .. 2^60, one piece at a time
          const uint32_t b = by_nc.div(row);
          Piece<T> q;
          q.load(x + (int64_t)b * s_b + (int64_t)(row - b * by_nc.d) * s_nc + (int64_t)k * 16, false);
          uint32_t c[4] = {0u, 0u, 0u, 0u};
#pragma unroll
          for (int i = 0; i < 16; i += 2) {
            const float t0 = quot(q.at(i)), t1 = quot(q.at(i + 1));
            c[i >> 2] |= (f == 0 ? quant2<0>(t0, t1) : f == 1 ? quant2<1>(t0, t1) : quant2<2>(t0, t1)) << (16 * (i >> 1 & 1));
          }
          dst[k] = make_uint4(c[0], c[1], c[2], c[3]);
        }
      }
    }
    row = row_next;                                                     // (rows + a step fit 32 bits: rows_spread)
  }
}

// ---------------------------------------------------------------- quantize + transpose
// Storage [c][nc] (nc contiguous) -> codes [nc][ldc] and optional bf16 copies [nc][c].
// A 64(c) x 64(nc) tile goes through shared memory.
// scale(output row, whether this thread also stores it): the row's Eq. 1 scale.
template <typename T, int FMT, typename Scale>
__device__ __forceinline__ void transpose_general(const T* __restrict__ x, int64_t nc, int64_t c, int64_t s_c, int64_t s_b,
                                                  Scale scale, uint8_t* __restrict__ codes, int64_t ldc,
                                                  __nv_bfloat16* __restrict__ abs_copy, __nv_bfloat16* __restrict__ kmaj_copy,
                                                  const Rounding& rnd, float (&tile)[64][65], const uint3 at) {
  const int64_t b = at.z;
  const int64_t c0 = (int64_t)at.y * 64, n0 = (int64_t)at.x * 64;
  const T* base = x + b * s_b;
  const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;    // 8 column-chunks x 32 rows
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const int rr = ty + it * 32;
    const int64_t cc = c0 + rr, nn = n0 + tx * 8;
    Vec8 v;
    if (cc < c && nn + 8 <= nc) v = Loader<T>::load8(base + cc * s_c + nn);
    else {
#pragma unroll
      for (int j = 0; j < 8; ++j)
        v.v[j] = (cc < c && nn + j < nc) ? Loader<T>::load1(base, cc * s_c + nn + j) : 0.f;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) tile[rr][tx * 8 + j] = v.v[j];
  }
  __syncthreads();
  // output: row n (64 of them), 64 contraction entries = 8 chunks of 8
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const int nrow = ty + it * 32;
    const int64_t nn = n0 + nrow;
    if (nn >= nc) continue;
    const int64_t k0 = c0 + tx * 8;
    if (k0 >= ldc) continue;
    Vec8 v;
#pragma unroll
    for (int j = 0; j < 8; ++j) v.v[j] = tile[tx * 8 + j][nrow];
    const Quotient quot(scale(b * nc + nn, at.y == 0 && tx == 0));
    const int64_t orow = b * nc + nn;
    *reinterpret_cast<uint2*>(codes + orow * ldc + k0) =
        rnd.stochastic ? quant8_sr<FMT>(v, quot, rnd, (uint64_t)orow * (uint64_t)c + (uint64_t)k0)
                       : quant8<FMT>(v, quot);
    if (abs_copy || kmaj_copy) {
      if (k0 + 8 <= c && (c & 7) == 0) {
        if (abs_copy) *reinterpret_cast<uint4*>(abs_copy + orow * c + k0) = abs_bf16x8(v);
        if (kmaj_copy) *reinterpret_cast<uint4*>(kmaj_copy + orow * c + k0) = to_bf16x8(v);
      } else {
        for (int j = 0; j < 8 && k0 + j < c; ++j) {
          if (abs_copy) abs_copy[orow * c + k0 + j] = __float2bfloat16_rn(fabsf(v.v[j]));
          if (kmaj_copy) kmaj_copy[orow * c + k0 + j] = __float2bfloat16_rn(v.v[j]);
        }
      }
    }
  }
}

template <typename T, int FMT>
__global__ void __launch_bounds__(kThreads)
quantize_transpose_kernel(const T* __restrict__ x, int64_t nc, int64_t c, int64_t s_c, int64_t s_b,
                          const DeltaSrc ds, uint8_t* __restrict__ codes, int64_t ldc,
                          __nv_bfloat16* __restrict__ abs_copy, __nv_bfloat16* __restrict__ kmaj_copy,
                          const Rounding rnd) {
  pdl_prologue();
  __shared__ float tile[64][65];     // +1 column spreads the transposed accesses over the banks
  const float d_tensor = ds.per_channel
                             ? 0.f
                             : ds.get(0, blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0);
  transpose_general<T, FMT>(x, nc, c, s_c, s_b, [&](int64_t row, bool writer) { return ds.per_channel ? ds.get(row, writer) : d_tensor; },
                            codes, ldc, abs_copy, kmaj_copy, rnd, tile, blockIdx);
}

// ---------------------------------------------------------------- quantize + transpose, bf16 fast path
// Storage [c][nc] (nc contiguous, bf16) with c a multiple of 32 and nc even.  A thread owns two
// adjacent columns and 32 consecutive contraction rows: it issues its 32 four-byte loads (each
// warp-wide load is one 128-byte row segment) before using any, then writes 32 bytes of codes
// and 64 bytes of each bf16 copy per column - whole sectors, no shared memory, no barrier.
// Block = 8 warps = 64 columns x 256 rows.
template <int FMT>
__global__ void __launch_bounds__(kThreads)
quantize_transpose_bf16_kernel(const __nv_bfloat16* __restrict__ x, int64_t nc, int64_t c, int64_t s_c,
                               int64_t s_b, const DeltaSrc ds, uint8_t* __restrict__ codes, int64_t ldc,
                               __nv_bfloat16* __restrict__ abs_copy, __nv_bfloat16* __restrict__ kmaj_copy) {
  pdl_prologue();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t b = blockIdx.z;
  const int64_t n = ((int64_t)blockIdx.x * 32 + lane) * 2;                 // first of this thread's two columns
  const int64_t k0 = ((int64_t)blockIdx.y * 8 + warp) * 32;                // first contraction row
  const float d_tensor =
      ds.per_channel ? 0.f : ds.get(0, blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0);
  if (n >= nc || k0 >= c) return;
  const uint32_t* src = reinterpret_cast<const uint32_t*>(x + b * s_b + k0 * s_c + n);
  const int64_t step = s_c >> 1;                                           // row stride in 32-bit words
  uint32_t w[32];
#pragma unroll
  for (int r = 0; r < 32; ++r) w[r] = __ldg(src + r * step);
#pragma unroll
  for (int col = 0; col < 2; ++col) {
    const int64_t orow = b * nc + n + col;
    const float dv = ds.per_channel ? ds.get(orow, k0 == 0) : d_tensor;
    // this column's 32 values as 16 words of two bf16 each
    uint32_t pw[16];
#pragma unroll
    for (int j = 0; j < 16; ++j)
      pw[j] = col == 0 ? __byte_perm(w[2 * j], w[2 * j + 1], 0x5410) : __byte_perm(w[2 * j], w[2 * j + 1], 0x7632);
    uint4* cdst = reinterpret_cast<uint4*>(codes + orow * ldc + k0);
    if (QuotientPair::serves(dv)) {
      const QuotientPair qp(dv);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint4 a = make_uint4(pw[8 * h], pw[8 * h + 1], pw[8 * h + 2], pw[8 * h + 3]);
        const uint4 bb = make_uint4(pw[8 * h + 4], pw[8 * h + 5], pw[8 * h + 6], pw[8 * h + 7]);
        cdst[h] = ds.from_amax ? quant_bf16x16<FMT, false>(a, bb, qp) : quant_bf16x16<FMT, true>(a, bb, qp);
      }
    } else {
      const Quotient quot(dv);
      uint32_t cw[8];
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        Vec8 f;
#pragma unroll
        for (int j = 0; j < 4; ++j) { f.v[2 * j] = bf16_lo(pw[4 * g + j]); f.v[2 * j + 1] = bf16_hi(pw[4 * g + j]); }
        const uint2 q = quant8<FMT>(f, quot);
        cw[2 * g] = q.x; cw[2 * g + 1] = q.y;
      }
      cdst[0] = make_uint4(cw[0], cw[1], cw[2], cw[3]);
      cdst[1] = make_uint4(cw[4], cw[5], cw[6], cw[7]);
    }
    if (abs_copy || kmaj_copy) {
      if (kmaj_copy) {
        uint4* d = reinterpret_cast<uint4*>(kmaj_copy + orow * c + k0);
#pragma unroll
        for (int j = 0; j < 4; ++j) d[j] = make_uint4(pw[4 * j], pw[4 * j + 1], pw[4 * j + 2], pw[4 * j + 3]);
      }
      if (abs_copy) {
        const uint32_t m = 0x7fff7fffu;
        uint4* d = reinterpret_cast<uint4*>(abs_copy + orow * c + k0);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          d[j] = make_uint4(pw[4 * j] & m, pw[4 * j + 1] & m, pw[4 * j + 2] & m, pw[4 * j + 3] & m);
      }
    }
  }
}

// ---------------------------------------------------------------- quantize in storage order, a scale per column
// Storage [c][nc] (nc contiguous, bf16), a scale per column, codes in the same order: [c] rows of ldn bytes, every format
// in MASK.  A block takes 64, 128 or 256 columns (8 << lane_bits) x a run of rows; its threads first make a column's scales each
// (maximum bits from `bits`), then a thread takes eight columns of four rows at a time.  Bound by HBM.  Blocks of 256 columns
// whatever the operand's width leave most lanes of a narrow one without columns; us, transposed / 256 columns a block / so:
// 512 x 64 x 512 in a batch of 256, one format 15.9 / 27.9 / 16.3, three formats 30 (three launches) / 62 / 25; 40 columns of 128
// in a batch of 512 8.6 / 12.8 / 7.8 and 24 / 30.5 / 13.3.
struct ColScales { float recip[256], ndelta[256]; };      // recip 0: outside the range of the two-wide quotient
template <int MASK, typename Bits>
__device__ __forceinline__ void quantize_cols(const __nv_bfloat16* __restrict__ x, int64_t nc, int64_t s_c, int64_t row0, int64_t row1,
                                              int64_t col_block, int lane_bits, Bits bits, bool writer, const MultiOut& o,
                                              int64_t delta_at, int64_t code_row0, int64_t ldn, ColScales* sc) {
  const int cols = 8 << lane_bits, rows_at_once = 8 * (32 >> lane_bits);    // columns of the block, rows that its lanes cover
  if ((int)threadIdx.x < cols) {
    const int64_t col = col_block * cols + threadIdx.x;
    const uint32_t m = col < nc ? bits(col) : 0u;
    int k = 0;
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      if (!(MASK & (1 << f))) continue;
      const float d = m == 0 ? 1.0f : __fdiv_rn(__uint_as_float(m), fmt_qmax(f));
      sc[k].recip[threadIdx.x] = QuotientPair::serves(d) ? __frcp_rn(d) : 0.f;
      sc[k].ndelta[threadIdx.x] = -d;
      ++k;
      if (writer && col < nc) {
        o.delta_out[f][delta_at + col] = d;
        if (m >= 0x7f800000u && o.err_word[f]) atomicOr(o.err_word[f], QM_DEVERR_NONFINITE);
      }
    }
  }
  __syncthreads();
  const int group = threadIdx.x & ((1 << lane_bits) - 1);              // of eight columns
  const int64_t col0 = col_block * cols + group * 8;
  if (col0 >= nc) return;
  const int live = nc - col0 < 8 ? (int)(nc - col0) : 8;
  const __nv_bfloat16* base = x + col0;
  for (int64_t r = row0 + (threadIdx.x >> lane_bits); r < row1; r += 4 * rows_at_once) {
    uint4 w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t row = r + u * rows_at_once < row1 ? r + u * rows_at_once : r;          // repeats are not written
      if (live == 8) {
        w[u] = __ldg(reinterpret_cast<const uint4*>(base + row * s_c));
      } else {
        const unsigned short* e = reinterpret_cast<const unsigned short*>(base + row * s_c);
        uint32_t h[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) h[j] = j < live ? (uint32_t)__ldg(e + j) : 0u;
        w[u] = make_uint4(h[0] | h[1] << 16, h[2] | h[3] << 16, h[4] | h[5] << 16, h[6] | h[7] << 16);
      }
    }
    int k = 0;
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      if (!(MASK & (1 << f))) continue;
      const ColScales& cs = sc[k];
      ++k;
      float rc[8];
      uint64_t r2[4], n2[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        r2[j] = *reinterpret_cast<const uint64_t*>(&cs.recip[group * 8 + 2 * j]);
        n2[j] = *reinterpret_cast<const uint64_t*>(&cs.ndelta[group * 8 + 2 * j]);
        asm("mov.b64 {%0, %1}, %2;" : "=f"(rc[2 * j]), "=f"(rc[2 * j + 1]) : "l"(r2[j]));
      }
      bool served = true;
#pragma unroll
      for (int j = 0; j < 8; ++j) served &= rc[j] != 0.f;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (r + u * rows_at_once >= row1) break;
        const uint32_t pw[4] = {w[u].x, w[u].y, w[u].z, w[u].w};
        uint2 q;
        if (served) {
          uint32_t h[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const QuotientPair qp(r2[j], n2[j]);
            h[j] = (f == 0 ? quant_bf16_pair<0>(pw[j], qp) : f == 1 ? quant_bf16_pair<1>(pw[j], qp) : quant_bf16_pair<2>(pw[j], qp)) & 0xffffu;
          }
          q = make_uint2(h[0] | h[1] << 16, h[2] | h[3] << 16);
        } else {
          uint32_t h[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float t0 = Quotient(-cs.ndelta[group * 8 + 2 * j])(bf16_lo(pw[j])), t1 = Quotient(-cs.ndelta[group * 8 + 2 * j + 1])(bf16_hi(pw[j]));
            h[j] = f == 0 ? quant2<0>(t0, t1) : f == 1 ? quant2<1>(t0, t1) : quant2<2>(t0, t1);
          }
          q = make_uint2(h[0] | h[1] << 16, h[2] | h[3] << 16);
        }
        *reinterpret_cast<uint2*>(o.codes[f] + (code_row0 + r + u * rows_at_once) * ldn + col0) = q;
      }
    }
  }
}

template <int MASK>
__global__ void __launch_bounds__(kThreads)
quantize_cols_kernel(const __nv_bfloat16* __restrict__ x, int64_t nc, int64_t c, int64_t s_c, int64_t s_b, int64_t rows_per_block,
                     int lane_bits, const uint32_t* __restrict__ amax, const MultiOut o, int64_t ldn) {
  pdl_prologue();
  __shared__ __align__(16) ColScales sc[(MASK & 1) + (MASK >> 1 & 1) + (MASK >> 2 & 1)];
  const int64_t b = blockIdx.z, row0 = (int64_t)blockIdx.y * rows_per_block, row1 = min(c, row0 + rows_per_block);
  quantize_cols<MASK>(x + b * s_b, nc, s_c, row0, row1, blockIdx.x, lane_bits, [&](int64_t col) { return __ldg(amax + b * nc + col); },
                      blockIdx.y == 0, o, b * nc, b * c, ldn, sc);
}

// Eight columns a lane: as many lanes to a row as leave the fewest of them without columns, the most if several do (wide
// operands are as fast in narrow blocks: 3078 columns of 2032 in three formats, the whole batch 96 us in blocks of 256, 93 of 64).
__host__ inline int col_lane_bits(int64_t nc) {
  int best = 5;
  for (int bits = 4; bits >= 3; --bits) {
    const int64_t w = 8 << bits, wb = 8 << best;
    if ((nc + w - 1) / w * w < (nc + wb - 1) / wb * wb) best = bits;
  }
  return best;
}

// ---------------------------------------------------------------- both operands of a probe in two launches
// A probe of modest operands is bound by its chain of launches, not by what they do: clear, max|x| and
// quantize for one operand, the same for the other, products.  Here one kernel takes the maxima of both
// operands and one quantizes both, so that the operands run side by side and the chain is three launches
// long.  The maxima are partial ones, stored (not combined by atomics), so nothing has to be cleared first:
//   one scale per tensor:      a maximum per block of the first kernel (at most kPairBlocks);
//   one per strided channel:   a maximum per column and slice of the contraction (at most kPairSlices);
//   one per contiguous row:    none, the second kernel reduces a row itself.
constexpr int kPairBlocks = 256, kPairSlices = 8;
constexpr int kPairColRows = 64;          // rows of a block of kPairCols
enum { kPairChunks = 0, kPairRows = 1, kPairTiles = 2, kPairGeneral = 3, kPairCols = 4 };

struct PairOperand {
  View v;
  int32_t fmt, per_channel;
  int32_t blocks_max, n_partial;          // blocks of the first kernel; partial maxima per scale
  int32_t blocks_quant, path;             // blocks of the second kernel, and how it walks the operand
  uint32_t gx, gy;                        // tiles: column tiles, contraction tiles
  uint32_t max_cols;                      // one scale per strided channel: blocks of 64 columns
  int32_t col_lane_bits;                  // kPairCols: see quantize_cols
  uint32_t groups_per_line, total_groups, lines;   // the tensor as lines of contiguous groups of eight; lines per batch element
  FastDiv by_groups, by_lines, by_chunks, by_nc, by_gx, by_gy, by_max_cols;
  uint32_t* partial;
  float* delta;
  uint8_t* codes;
  Rounding rnd;
};
struct PairArgs {
  PairOperand op[2];
  uint32_t* control;                      // cleared by the first kernel; its first word takes the error flags
  uint32_t control_words;
  uint32_t clusters[2];                   // the one-launch form: clusters of each operand
};

// Eight elements as loaded, and running maxima of their magnitudes, element by element (bf16: two to a word).
template <typename T> struct Raw8;
template <> struct Raw8<__nv_bfloat16> {
  static constexpr int kWords = 4;
  uint32_t w[4];
  __device__ __forceinline__ void load(const __nv_bfloat16* p, int live) {
    if (live >= 8) {
      const uint4 q = __ldg(reinterpret_cast<const uint4*>(p));
      w[0] = q.x; w[1] = q.y; w[2] = q.z; w[3] = q.w;
    } else {
      const unsigned short* e = reinterpret_cast<const unsigned short*>(p);
#pragma unroll
      for (int j = 0; j < 4; ++j) w[j] = (2 * j < live ? (uint32_t)__ldg(e + 2 * j) : 0u) | (2 * j + 1 < live ? (uint32_t)__ldg(e + 2 * j + 1) << 16 : 0u);
    }
  }
  // what lies beyond `live` elements (from 1 on) is zero
  __device__ __forceinline__ void keep(uint32_t live) {
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j) w[j] = 2 * j + 1 < live ? w[j] : 2 * j < live ? w[j] & 0xffffu : 0u;
  }
  static __device__ __forceinline__ uint32_t upper(uint32_t m, uint32_t x) { return __vmaxu2(m, x & 0x7fff7fffu); }
  static __device__ __forceinline__ uint32_t both(uint32_t m, uint32_t n) { return __vmaxu2(m, n); }
  // element j of the maxima as an fp32 pattern
  static __device__ __forceinline__ uint32_t element(const uint32_t* m, int j) { return j & 1 ? m[j >> 1] & 0xffff0000u : m[j >> 1] << 16; }
};
template <> struct Raw8<float> {
  static constexpr int kWords = 8;
  uint32_t w[8];
  __device__ __forceinline__ void load(const float* p, int live) {
    if (live >= 8) {
      const uint4 q = __ldg(reinterpret_cast<const uint4*>(p)), r = __ldg(reinterpret_cast<const uint4*>(p) + 1);
      w[0] = q.x; w[1] = q.y; w[2] = q.z; w[3] = q.w; w[4] = r.x; w[5] = r.y; w[6] = r.z; w[7] = r.w;
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) w[j] = j < live ? __float_as_uint(__ldg(p + j)) : 0u;
    }
  }
  __device__ __forceinline__ void keep(uint32_t live) {
#pragma unroll
    for (uint32_t j = 0; j < 8; ++j) w[j] = j < live ? w[j] : 0u;
  }
  static __device__ __forceinline__ uint32_t upper(uint32_t m, uint32_t x) { return max(m, x & 0x7fffffffu); }
  static __device__ __forceinline__ uint32_t both(uint32_t m, uint32_t n) { return max(m, n); }
  static __device__ __forceinline__ uint32_t element(const uint32_t* m, int j) { return m[j]; }
};

// max|x| of every blocks-th piece of the tensor; valid in warp 0.  AHEAD: loads of a thread on their way together (a round trip
// is what these loops wait for).
template <typename T, int AHEAD>
__device__ __forceinline__ uint32_t pair_tensor_max(const PairOperand& o, uint32_t block, uint32_t blocks) {
  using Raw = Raw8<T>;
  const View& v = o.v;
  const T* x = static_cast<const T*>(v.data);
  const bool along_c = v.s_c == 1;
  const int64_t inner = along_c ? v.c : v.nc, line_stride = along_c ? v.s_nc : v.s_c;
  const uint32_t stride = blocks * kThreads;
  uint32_t acc[Raw::kWords] = {};
  auto group = [&](uint32_t g, uint32_t* k) {
    const uint32_t line = o.by_groups.div(g), b = o.by_lines.div(line);
    *k = (g - line * o.groups_per_line) * 8;
    return x + (int64_t)b * v.s_b + (int64_t)(line - b * o.lines) * line_stride + *k;
  };
  auto fold = [&](const Raw& w) {
#pragma unroll
    for (int j = 0; j < Raw::kWords; ++j) acc[j] = Raw::upper(acc[j], w.w[j]);
  };
  // A line's last group is loaded whole as well and what lies beyond the line is taken out (strides are multiples of eight, so it belongs to
  // the tensor's span; but for the very last group): a branch between the loads makes each of them a round trip of its own
  auto pass = [&](auto whole, uint32_t groups) {
    for (uint32_t g0 = block * kThreads + threadIdx.x; g0 < groups; g0 += AHEAD * stride) {
      Raw w[AHEAD];
      uint32_t k[AHEAD];
#pragma unroll
      for (int u = 0; u < AHEAD; ++u) w[u].load(group(g0 + u * stride < groups ? g0 + u * stride : g0, &k[u]), 8);      // repeats change no maximum
#pragma unroll
      for (int u = 0; u < AHEAD; ++u) {
        if (!decltype(whole)::value) w[u].keep((uint32_t)inner - k[u]);
        fold(w[u]);
      }
    }
  };
  if ((inner & 7) == 0) {
    pass(std::true_type{}, o.total_groups);
  } else {
    pass(std::false_type{}, o.total_groups - 1);
    if (block == blocks - 1 && threadIdx.x == kThreads - 1) {
      Raw w;
      uint32_t k;
      const T* const p = group(o.total_groups - 1, &k);
      w.load(p, (int)((uint32_t)inner - k));
      fold(w);
    }
  }
#pragma unroll
  for (int j = 1; j < Raw::kWords; ++j) acc[0] = Raw::both(acc[0], acc[j]);
  return block_max(max(Raw::element(acc, 0), Raw::kWords == 4 ? Raw::element(acc, 1) : 0u));
}
// The maxima of 8 << lane_bits columns from `first` on of batch element b over rows r0 .. r1 - 1, left in s: thread t < 8 <<
// lane_bits returns that of column first + t.
template <typename T, int AHEAD>
__device__ __forceinline__ uint32_t pair_column_max(const PairOperand& o, int64_t b, int64_t first, int lane_bits, int64_t r0, int64_t r1,
                                                    uint32_t* s) {
  using Raw = Raw8<T>;
  const View& v = o.v;
  const int cols = 8 << lane_bits, rows_at_once = kThreads >> lane_bits;
  const int tx = threadIdx.x & ((1 << lane_bits) - 1), ty = threadIdx.x >> lane_bits;
  const int64_t col0 = first + tx * 8;
  const T* base = static_cast<const T*>(v.data) + b * v.s_b + col0;
  uint32_t acc[Raw::kWords] = {};
  if (col0 < v.nc) {
    const int live = v.nc - col0 < 8 ? (int)(v.nc - col0) : 8;
    for (int64_t r = r0 + ty; r < r1; r += AHEAD * rows_at_once) {
      Raw w[AHEAD];
#pragma unroll
      for (int u = 0; u < AHEAD; ++u) {
        const int64_t row = r + u * rows_at_once < r1 ? r + u * rows_at_once : r;
        w[u].load(base + row * v.s_c, live);
      }
#pragma unroll
      for (int u = 0; u < AHEAD; ++u)
#pragma unroll
        for (int j = 0; j < Raw::kWords; ++j) acc[j] = Raw::upper(acc[j], w[u].w[j]);
    }
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) s[ty * cols + tx * 8 + j] = Raw::element(acc, j);
  __syncthreads();
  uint32_t m = 0;
  if ((int)threadIdx.x < cols)
    for (int j = 0; j < rows_at_once; ++j) m = max(m, s[j * cols + threadIdx.x]);
  return m;
}

template <typename T>
__device__ __forceinline__ void pair_max(const PairOperand& o, uint32_t block, uint32_t* s) {
  const View& v = o.v;
  if (!o.per_channel) {
    const uint32_t m = pair_tensor_max<T, 4>(o, block, (uint32_t)o.blocks_max);
    if (threadIdx.x == 0) o.partial[block] = m;
    return;
  }
  // a column each: 64 columns of one batch element, one slice of the contraction
  const uint32_t slice = block % (uint32_t)o.n_partial, rest = block / (uint32_t)o.n_partial;
  const uint32_t b = o.by_max_cols.div(rest), cb = rest - b * o.max_cols;
  const int64_t per = (v.c + o.n_partial - 1) / o.n_partial, r0 = slice * per, r1 = r0 + per < v.c ? r0 + per : v.c;
  const uint32_t m = pair_column_max<T, 4>(o, b, (int64_t)cb * 64, 3, r0, r1, s);
  const int64_t col = (int64_t)cb * 64 + threadIdx.x;
  if (threadIdx.x < 64 && col < v.nc) o.partial[((int64_t)slice * v.batch + b) * v.nc + col] = m;
}

__global__ void __launch_bounds__(kThreads) pair_max_kernel(const PairArgs a) {
  pdl_prologue();
  __shared__ uint32_t s[32 * 64];
  if (blockIdx.x == 0 && threadIdx.x < a.control_words) a.control[threadIdx.x] = 0u;
  const bool right = blockIdx.x >= (uint32_t)a.op[0].blocks_max;
  const PairOperand& o = right ? a.op[1] : a.op[0];
  const uint32_t block = right ? blockIdx.x - a.op[0].blocks_max : blockIdx.x;
  if (block >= (uint32_t)o.blocks_max) return;          // (where neither operand has maxima one block still clears)
  if (o.v.dtype == QM_DT_BF16) pair_max<__nv_bfloat16>(o, block, s);
  else pair_max<float>(o, block, s);
}

// The scale of an output row (0: of the tensor) from its max|x|; the thread that is told to stores it.
template <int FMT>
__device__ __forceinline__ float pair_scale(const PairOperand& o, uint32_t bits, int64_t at, bool writer, uint32_t* err) {
  const float d = bits == 0 ? 1.0f : __fdiv_rn(__uint_as_float(bits), fmt_qmax(FMT));
  if (writer) {
    o.delta[at] = d;
    if (bits >= 0x7f800000u) atomicOr(err, QM_DEVERR_NONFINITE);
  }
  return d;
}

// The codes of a block of the second kernel, whatever takes its maxima: d_tensor where there is one scale, else
// col_bits(row of the output) its max|x|.  SR_TILES: strided bf16 may be rounded stochastically.
template <typename T, int FMT, bool SR_TILES, typename Bits>
__device__ __forceinline__ void pair_codes(const PairOperand& o, uint32_t* err, uint32_t block, uint4* smem, float d_tensor, Bits col_bits) {
  const View& v = o.v;
  const T* x = static_cast<const T*>(v.data);
  const int64_t ldc = (v.c + 15) & ~(int64_t)15;
  auto scale = [&](int64_t row, bool writer) {
    return o.per_channel ? pair_scale<FMT>(o, col_bits(row), row, writer, err) : d_tensor;
  };
  if (o.path == kPairChunks) {              // contiguous contraction: sixteen elements per thread
    const uint32_t chunks = (uint32_t)(ldc >> 4), i = block * kThreads + threadIdx.x;
    if (i >= (uint32_t)(v.nc * v.batch) * chunks) return;
    const uint32_t row = o.by_chunks.div(i), b = o.by_nc.div(row);
    const int64_t k0 = (int64_t)(i - row * chunks) * 16;
    const T* p = x + (int64_t)b * v.s_b + (int64_t)(row - b * (uint32_t)v.nc) * v.s_nc + k0;
    uint4* dst = reinterpret_cast<uint4*>(o.codes + (int64_t)row * ldc + k0);
    const uint64_t number = (uint64_t)row * (uint64_t)v.c + (uint64_t)k0;
    if (sizeof(T) == 2 && k0 + 16 <= v.c && QuotientPair::serves(d_tensor) && (!o.rnd.stochastic || (number & 3) == 0)) {
      const uint4 lo = __ldg(reinterpret_cast<const uint4*>(p)), hi = __ldg(reinterpret_cast<const uint4*>(p) + 1);
      const QuotientPair qp(d_tensor);
      *dst = o.rnd.stochastic ? quant_bf16x16_sr<FMT, false>(lo, hi, qp, o.rnd, number) : quant_bf16x16<FMT>(lo, hi, qp);
      return;
    }
    const Quotient quot(d_tensor);
    uint2 q[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      Vec8 w;
      if (k0 + 8 * h + 8 <= v.c) {
        w = Loader<T>::load8(p + 8 * h);
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) w.v[j] = k0 + 8 * h + j < v.c ? Loader<T>::load1(p, 8 * h + j) : 0.f;
      }
      q[h] = o.rnd.stochastic ? quant8_sr<FMT>(w, quot, o.rnd, number + 8 * h) : quant8<FMT>(w, quot);
    }
    *dst = make_uint4(q[0].x, q[0].y, q[1].x, q[1].y);
    return;
  }
  // strided contraction: tiles
  const uint32_t rest = o.by_gx.div(block), bz = o.by_gy.div(rest);
  const uint3 at = make_uint3(block - rest * o.gx, rest - bz * o.gy, bz);
  if constexpr (sizeof(T) == 2) {
    if (o.path == kPairCols) {              // codes in storage order, a scale per column
      MultiOut out{};
      out.codes[FMT] = o.codes; out.delta_out[FMT] = o.delta; out.err_word[FMT] = err;
      const int64_t row0 = (int64_t)at.y * kPairColRows, row1 = row0 + kPairColRows < v.c ? row0 + kPairColRows : v.c;
      auto bits = [&](int64_t col) { return col_bits((int64_t)at.z * v.nc + col); };
      quantize_cols<1 << FMT>(x + (int64_t)at.z * v.s_b, v.nc, v.s_c, row0, row1, at.x, o.col_lane_bits, bits, at.y == 0, out, (int64_t)at.z * v.nc,
                              (int64_t)at.z * v.c, (v.nc + 15) & ~(int64_t)15, reinterpret_cast<ColScales*>(smem));
      return;
    }
  }
  if (o.path == kPairGeneral) {
    transpose_general<T, FMT>(x, v.nc, v.c, v.s_c, v.s_b, scale, o.codes, ldc, nullptr, nullptr, o.rnd,
                              *reinterpret_cast<float(*)[64][65]>(smem), at);
    return;
  }
  if constexpr (sizeof(T) == 2) {
    const int64_t col = (int64_t)at.x * 64 + 2 * (threadIdx.x & 31), orow = (int64_t)at.z * v.nc + col;
    const bool writer = at.y == 0 && threadIdx.x < 32;
    float d_lo[3] = {1.f, 1.f, 1.f}, d_hi[3] = {1.f, 1.f, 1.f};
    if (col < v.nc) d_lo[FMT] = scale(orow, writer);
    if (col + 1 < v.nc) d_hi[FMT] = scale(orow + 1, writer);
    uint8_t* const cd[3] = {o.codes, o.codes, o.codes};
    if (SR_TILES && o.rnd.stochastic) transpose_tile<1 << FMT, false, true, SR_TILES>(x, v.nc, v.c, v.s_c, v.s_b, d_lo, d_hi, cd, ldc, nullptr, smem, at, o.rnd);
    else transpose_tile<1 << FMT, false, true, false>(x, v.nc, v.c, v.s_c, v.s_b, d_lo, d_hi, cd, ldc, nullptr, smem, at);
  }
}

template <typename T, int FMT>
__device__ __forceinline__ void pair_quantize(const PairOperand& o, uint32_t* err, uint32_t block, uint4* smem) {
  const View& v = o.v;
  if (o.path == kPairRows) {
    scale_quantize_rows<T, FMT, 32>(static_cast<const T*>(v.data), v.nc, v.c, v.s_nc, v.batch, v.s_b, fmt_qmax(FMT), o.delta, o.codes,
                                    (v.c + 15) & ~(int64_t)15, nullptr, err, block);
    return;
  }
  float d_tensor = 1.f;
  if (!o.per_channel) {
    uint32_t m = 0;
    for (int i = threadIdx.x & 31; i < o.n_partial; i += 32) m = max(m, __ldg(o.partial + i));
    d_tensor = pair_scale<FMT>(o, warp_max(m), 0, block == 0 && threadIdx.x == 0, err);
  }
  pair_codes<T, FMT, true>(o, err, block, smem, d_tensor, [&](int64_t row) {
    uint32_t m = 0;
    for (int i = 0; i < o.n_partial; ++i) m = max(m, __ldg(o.partial + (int64_t)i * v.batch * v.nc + row));
    return m;
  });
}

// F0, F1: the operands' formats; T: their element type.
template <typename T, int F0, int F1>
__global__ void __launch_bounds__(kThreads) pair_quantize_kernel(const PairArgs a) {
  pdl_prologue();
  __shared__ uint4 smem[TileSmem<1>::kVec];             // a bf16 tile with codes and copy, or a 64 x 65 fp32 tile
  static_assert(sizeof(float) * 64 * 65 <= sizeof(uint4) * TileSmem<1>::kVec, "the general tile has to fit");
  if (blockIdx.x < (uint32_t)a.op[0].blocks_quant) pair_quantize<T, F0>(a.op[0], a.control, blockIdx.x, smem);
  else pair_quantize<T, F1>(a.op[1], a.control, blockIdx.x - a.op[0].blocks_quant, smem);
}

// ---------------------------------------------------------------- the tensors of a batch in two launches
// Dense bf16 tensors under one scale each: max|x| of all of them in one launch, the codes of all their formats in another.  A
// launch for each tensor and step, spread over streams, is bound by its submission and by 3 to 4 us a launch where the tensors are
// small: the four products of a BERT-base layer in two formats (six tensors, 46 MB) took 40 us to prepare in twelve launches.
struct ManyMax { const uint8_t* x; uint64_t n_vec; uint32_t* amax; uint32_t block0; };      // n_vec: 32-byte vectors
struct ManyCodes {
  const uint8_t* x; const uint32_t* amax;
  float* delta[3]; uint32_t* err[3]; uint4* codes[3];         // by format; codes null: not asked for
  uint32_t chunks, block0;                                   // chunks: of 16 elements
};
template <typename E> struct ManyList { int n; E e[kManyTensors]; };
static_assert(sizeof(ManyList<ManyCodes>) <= 4096, "kernel parameters");
constexpr int kManyAhead = 4;              // 32-byte loads of a thread on their way together

template <typename E>
__device__ __forceinline__ int many_entry(const ManyList<E>& l, uint32_t block) {
  int i = 0;
  while (i + 1 < l.n && block >= l.e[i + 1].block0) ++i;
  return i;
}

__global__ void __launch_bounds__(kThreads) absmax_many_kernel(const __grid_constant__ ManyList<ManyMax> l) {
  const ManyMax e = l.e[many_entry(l, blockIdx.x)];
  pdl_prologue();
  const uint64_t i0 = (uint64_t)(blockIdx.x - e.block0) * (kThreads * kManyAhead) + threadIdx.x;
  Vec256 v[kManyAhead];
#pragma unroll
  for (int u = 0; u < kManyAhead; ++u) {
    const uint64_t i = i0 + u * kThreads;
    v[u] = ld256<false>(e.x + (i < e.n_vec ? i : e.n_vec - 1) * 32);          // repeats change no maximum
  }
  uint32_t m = 0;
  const uint32_t k = 0x7fff7fffu;
#pragma unroll
  for (int u = 0; u < kManyAhead; ++u) {
    const uint32_t a = __vmaxu2(__vmaxu2(v[u].lo.x & k, v[u].lo.y & k), __vmaxu2(v[u].lo.z & k, v[u].lo.w & k));
    const uint32_t b = __vmaxu2(__vmaxu2(v[u].hi.x & k, v[u].hi.y & k), __vmaxu2(v[u].hi.z & k, v[u].hi.w & k));
    m = __vmaxu2(m, __vmaxu2(a, b));
  }
  const uint32_t acc = block_max(max(m & 0xffffu, m >> 16) << 16);
  if (threadIdx.x == 0 && acc) atomicMax(e.amax, acc);
}

template <int CHUNKS>
__global__ void __launch_bounds__(kThreads) quantize_many_kernel(const __grid_constant__ ManyList<ManyCodes> l) {
  const uint32_t block = gridDim.x - 1 - blockIdx.x;         // backwards: what the maxima have read last is still in L2
  const ManyCodes& e = l.e[many_entry(l, block)];
  const uint32_t chunks = e.chunks, base = (block - e.block0) * (kThreads * CHUNKS) + threadIdx.x;
  const bool writer = block == e.block0 && threadIdx.x == 0;
  const uint8_t* const x = e.x;
  pdl_prologue();
  Vec256 w[CHUNKS];
#pragma unroll
  for (int u = 0; u < CHUNKS; ++u) {
    const uint32_t i = base + u * kThreads;
    w[u] = ld256<false>(x + 32 * (size_t)(i < chunks ? i : chunks - 1));
  }
  const uint32_t bits = __ldcg(e.amax);
  auto format = [&](auto fmt) {
    constexpr int F = decltype(fmt)::value;
    uint4* const codes = e.codes[F];
    if (!codes) return;
    const float d = bits == 0 ? 1.0f : __fdiv_rn(__uint_as_float(bits), fmt_qmax(F));
    if (writer) {
      *e.delta[F] = d;
      if (bits >= 0x7f800000u && e.err[F]) atomicOr(e.err[F], QM_DEVERR_NONFINITE);
    }
    if (QuotientPair::serves(d)) {
      const QuotientPair quot(d);
#pragma unroll
      for (int u = 0; u < CHUNKS; ++u)
        if (base + u * kThreads < chunks) codes[base + u * kThreads] = quant_bf16x16<F>(w[u].lo, w[u].hi, quot);
    } else {
      const Quotient quot(d);
#pragma unroll 1
      for (int u = 0; u < CHUNKS; ++u) {
        if (base + u * kThreads >= chunks) break;
        const Vec8 a = Loader<__nv_bfloat16>::load8(x + 32 * (size_t)(base + u * kThreads));
        const Vec8 b = Loader<__nv_bfloat16>::load8(x + 32 * (size_t)(base + u * kThreads) + 16);
        const uint2 p = quant8<F>(a, quot), q = quant8<F>(b, quot);
        codes[base + u * kThreads] = make_uint4(p.x, p.y, q.x, q.y);
      }
    }
  };
  format(std::integral_constant<int, 0>{});
  format(std::integral_constant<int, 1>{});
  format(std::integral_constant<int, 2>{});
}

// ---------------------------------------------------------------- both operands of a small probe in one launch
// Small enough that a cluster of eight blocks takes the maxima that it needs by itself, each block an eighth of them, and
// exchanges them through distributed shared memory: no block waits for another cluster, so the chain of a probe is one launch
// shorter.
//   one scale per tensor:      every cluster goes over the whole tensor (it comes from L2) and then makes its own share of the codes;
//   one per strided channel:   a cluster to a strip of columns, a block to an eighth of the contraction;
//   one per contiguous row:    a warp to a row, as in the two-launch form.
// Non-finite maxima are flagged in a byte for each block, always written: nobody could clear a common word ahead of
// all blocks.  They lie in the control block, which the products' last block reads.
constexpr int kOnceBlocks = 8;
// v into word `at` of the same array in block `rank` of the cluster
__device__ __forceinline__ void cluster_store(uint32_t* at, uint32_t rank, uint32_t v) {
  uint32_t to;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"((uint32_t)__cvta_generic_to_shared(at)), "r"(rank));
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(to), "r"(v) : "memory");
}

// s_max: a row of maxima from each block of the cluster, one of the tensor or one for each column of a strip.
template <typename T, int FMT>
__device__ __forceinline__ void pair_once(const PairOperand& o, uint32_t* err, uint32_t cluster, uint32_t clusters, uint32_t rank, uint4* smem,
                                          uint32_t (&s_max)[kOnceBlocks][64]) {
  constexpr int kAhead = 16 / sizeof(T);
  const View& v = o.v;
  if (o.path == kPairRows) {
    cluster_wait();
    const uint32_t block = cluster * kOnceBlocks + rank;
    if (block < (uint32_t)o.blocks_quant)
      scale_quantize_rows<T, FMT, 32>(static_cast<const T*>(v.data), v.nc, v.c, v.s_nc, v.batch, v.s_b, fmt_qmax(FMT), o.delta, o.codes,
                                      (v.c + 15) & ~(int64_t)15, nullptr, err, block);
    return;
  }
  auto cluster_max = [&](int i) {
    uint32_t m = 0;
#pragma unroll
    for (int k = 0; k < kOnceBlocks; ++k) m = max(m, s_max[k][i]);
    return m;
  };
  if (!o.per_channel) {
    const uint32_t m = pair_tensor_max<T, kAhead>(o, rank, kOnceBlocks);
    cluster_wait();                        // every block of the cluster has started
    if (threadIdx.x < kOnceBlocks) cluster_store(&s_max[rank][0], threadIdx.x, m);
    cluster_arrive();
    cluster_wait();
    const float d = pair_scale<FMT>(o, cluster_max(0), 0, cluster == 0 && rank == 0 && threadIdx.x == 0, err);
    for (uint32_t block = cluster * kOnceBlocks + rank; block < (uint32_t)o.blocks_quant; block += clusters * kOnceBlocks) {
      pair_codes<T, FMT, false>(o, err, block, smem, d, [](int64_t) { return 0u; });
      __syncthreads();                     // the tile's shared memory
    }
    return;
  }
  const uint32_t b = o.by_max_cols.div(cluster), strip = cluster - b * o.max_cols;
  constexpr int bits = 3;                  // strips of 64 columns
  const int64_t first = (int64_t)strip << (bits + 3);
  const int64_t per = (v.c + kOnceBlocks - 1) / kOnceBlocks, r0 = rank * per < v.c ? rank * per : v.c, r1 = r0 + per < v.c ? r0 + per : v.c;
  const uint32_t m = pair_column_max<T, kAhead>(o, b, first, bits, r0, r1, reinterpret_cast<uint32_t*>(smem));
  cluster_wait();
  if ((int)threadIdx.x < 8 << bits) {
#pragma unroll
    for (int k = 0; k < kOnceBlocks; ++k) cluster_store(&s_max[rank][threadIdx.x], k, m);
  }
  cluster_arrive();
  cluster_wait();
  if constexpr (sizeof(T) == 2) {
    if (o.path == kPairCols) {
      MultiOut out{};
      out.codes[FMT] = o.codes; out.delta_out[FMT] = o.delta; out.err_word[FMT] = err;
      quantize_cols<1 << FMT>(static_cast<const T*>(v.data) + (int64_t)b * v.s_b, v.nc, v.s_c, r0, r1, strip, bits,
                              [&](int64_t col) { return cluster_max((int)(col - first)); }, rank == 0, out, (int64_t)b * v.nc,
                              (int64_t)b * v.c, (v.nc + 15) & ~(int64_t)15, reinterpret_cast<ColScales*>(smem));
      return;
    }
  }
  for (uint32_t y = rank; y < o.gy; y += kOnceBlocks) {
    pair_codes<T, FMT, false>(o, err, (b * o.gy + y) * o.gx + strip, smem, 1.f, [&](int64_t row) { return cluster_max((int)(row - b * v.nc - first)); });
    __syncthreads();
  }
}

// T: the operands' element type.  INT: both INT8 (which goes with nothing else), else an FP8 format each, known at run time: six bodies to
// compile, where one for each pair of formats and side made twenty (this file 269 s, 146 so; the kernels as fast).
template <typename T, bool INT>
__global__ void __launch_bounds__(kThreads) pair_once_kernel(const PairArgs a) {
  __shared__ uint4 smem[TileSmem<1>::kVec];
  __shared__ uint32_t s_max[kOnceBlocks][64];
  __shared__ uint32_t s_err;
  cluster_arrive();
  if (threadIdx.x == 0) s_err = 0;
  __syncthreads();
  pdl_prologue();
  uint8_t* const flags = reinterpret_cast<uint8_t*>(a.control + kPrepareFlagWord);
  if (blockIdx.x == 0) {
    if (threadIdx.x < kPrepareFlagWord) a.control[threadIdx.x] = 0u;
    if (threadIdx.x >= gridDim.x && threadIdx.x < kPrepareFlags) flags[threadIdx.x] = 0;
  }
  const uint32_t cluster = blockIdx.x / kOnceBlocks, rank = blockIdx.x % kOnceBlocks;
  const bool right = cluster >= a.clusters[0];
  const PairOperand& o = right ? a.op[1] : a.op[0];
  const uint32_t at = right ? cluster - a.clusters[0] : cluster, clusters = a.clusters[right];
  if constexpr (INT) pair_once<T, QM_FMT_INT8>(o, &s_err, at, clusters, rank, smem, s_max);
  else if (o.fmt == QM_FMT_E4M3) pair_once<T, QM_FMT_E4M3>(o, &s_err, at, clusters, rank, smem, s_max);
  else pair_once<T, QM_FMT_E5M2>(o, &s_err, at, clusters, rank, smem, s_max);
  __syncthreads();
  if (threadIdx.x == 0) flags[blockIdx.x] = s_err ? 1 : 0;
}

// Clusters of an operand in the one-launch form; 0: not served.  Whole probes in a row, two launches / one, us.
//   One scale, read whole by every cluster: up to 256 KB of bf16 (512 x 512 x 256 17.4 / 16.5, 128 x 128 x 1024 21.6 / 20.8; of 384 KB 17.8 / 17.6
//   and 21.5 / 22.1, of 512 KB 17.3 / 17.7 and 22.0 / 22.9, of 1 MB 22.6 / 26.1), 512 KB of fp32, whose other form takes longer (512 x 128 x 256 24.1 /
//   21.9), and half of that where lines end inside a group of eight (131 columns, 128 KB 20.4 / 20.2, 192 KB 21.0 / 21.4, 256 KB 22.4 / 23.3).
//   A scale per strided column, an eighth of it to a block: columns up to 4 KB (bf16 64 x 64 x 2048 29.2 / 29.1, 512 x 512 x 2048 34.9 / 30.2, x 4096
//   41.8 / 43.3 and 48.3 / 45.8; fp32 64 x 64 x 1024 39.5 / 37.6, x 2048 65.2 / 67.2).
//   Strided bf16 rounded stochastically: not served (50 random probes: geometric mean 0.999; 56 x 82 x 1456 32.0 / 34.5, 66 x 220 x 32 19.1 / 21.2).
uint32_t once_clusters(const PairOperand& o, int elem) {
  const View& v = o.v;
  if (elem == 2 && o.rnd.stochastic && !v.c_contig()) return 0;
  const uint32_t clusters = (uint32_t)((o.blocks_quant + kOnceBlocks - 1) / kOnceBlocks);
  if (!o.per_channel) {
    const bool ragged = (v.c_contig() ? v.c : v.nc) & 7;
    return v.nc * v.c * v.batch * elem > ((elem == 2 ? 256 : 512) << 10) >> ragged ? 0 : clusters;
  }
  if (o.path == kPairRows) return clusters;
  return v.c * elem <= 4096 ? (uint32_t)(o.max_cols * v.batch) : 0;
}

int grid_for(int64_t work_items, int per_sm) {
  int64_t want = (work_items + kThreads - 1) / kThreads;
  int64_t cap = (int64_t)sm_count() * per_sm;
  return (int)(want < 1 ? 1 : (want < cap ? want : cap));
}

// max|x| over n dense elements: the 32-byte aligned middle by the 256-bit kernel, what is left at
// either end (less than 32 bytes each) by the general one.
template <typename T>
void absmax_dense(const T* p, int64_t n, uint32_t* amax, cudaStream_t s) {
  const uintptr_t a0 = reinterpret_cast<uintptr_t>(p), a1 = a0 + (uintptr_t)n * sizeof(T);
  const uintptr_t m0 = (a0 + 31) & ~(uintptr_t)31, m1 = a1 & ~(uintptr_t)31;
  if (m1 <= m0) {
    launch_pdl(absmax_tensor_kernel<T>, dim3(1), dim3(kThreads), 0, s, p, 1, n, n, FastDiv(), amax);
    return;
  }
  const uint64_t n_vec = (m1 - m0) / 32;
  const dim3 grid((unsigned)grid_for((int64_t)n_vec, 8));
  const uint8_t* mid = reinterpret_cast<const uint8_t*>(m0);
  if (m1 - m0 > (64u << 20))        // read once and far larger than what stays in L2: evict first
    launch_pdl(absmax_dense_kernel<T, 4, true>, grid, dim3(kThreads), 0, s, mid, n_vec, amax);
  else
    launch_pdl(absmax_dense_kernel<T, 4, false>, grid, dim3(kThreads), 0, s, mid, n_vec, amax);
  const int64_t head = (int64_t)((m0 - a0) / sizeof(T)), tail = (int64_t)((a1 - m1) / sizeof(T));
  if (head > 0) launch_pdl(absmax_tensor_kernel<T>, dim3(1), dim3(32), 0, s, p, 1, head, head, FastDiv(), amax);
  if (tail > 0) launch_pdl(absmax_tensor_kernel<T>, dim3(1), dim3(32), 0, s, p + (n - tail), 1, tail, tail, FastDiv(), amax);
}

// divisor of absmax_tensor_kernel for rows of n elements (of no use, and not used, below 8 or from 2^35 on)
FastDiv vec_div(int64_t n) { return n / 8 > 0 && n / 8 < (1ll << 32) ? FastDiv((uint32_t)(n / 8)) : FastDiv(); }

template <typename T>
qm_status absmax_t(const View& x, int gran, uint32_t* amax, cudaStream_t s) {
  const T* p = static_cast<const T*>(x.data);
  if (x.c_contig()) {
    if (gran == QM_GRAN_TENSOR) {
      const bool dense = x.s_nc == x.c && (x.batch == 1 || x.s_b == x.nc * x.c);
      const bool even = x.batch == 1 || x.s_b == x.nc * x.s_nc;
      if (dense) {
        const int64_t n = x.nc * x.batch * x.c;
        absmax_dense<T>(p, n, amax, s);
      } else if (even) {
        launch_pdl(absmax_tensor_kernel<T>, dim3(grid_for(x.nc * x.batch * x.c / 8 + 1, 8)), dim3(kThreads), 0, s, 
            p, x.nc * x.batch, x.c, x.s_nc, vec_div(x.c), amax);
      } else {
        for (int64_t b = 0; b < x.batch; ++b)
          launch_pdl(absmax_tensor_kernel<T>, dim3(grid_for(x.nc * x.c / 8 + 1, 8)), dim3(kThreads), 0, s, 
              p + b * x.s_b, x.nc, x.c, x.s_nc, vec_div(x.c), amax);
      }
    } else {
      const int64_t rows = x.nc * x.batch;
      const int64_t nvec = x.c / 8;
#define QM_ROWS(G)                                                                              \
  launch_pdl(absmax_rows_kernel<T, G>, dim3((unsigned)((rows * G + kThreads - 1) / kThreads)), dim3(kThreads), 0, s,  \
      p, x.nc, x.c, x.s_nc, x.batch, x.s_b, amax)
      if (nvec <= 4) QM_ROWS(4);
      else if (nvec <= 8) QM_ROWS(8);
      else if (nvec <= 16) QM_ROWS(16);
      else QM_ROWS(32);
#undef QM_ROWS
    }
  } else {
    if (gran == QM_GRAN_TENSOR) {
      // storage rows are the contracting index: walk them as rows of nc contiguous elements; the
      // rows of all batch elements form one run when the batch stride continues the row stride
      if (x.batch == 1 || x.s_b == x.c * x.s_c) {
        const bool dense = x.s_c == x.nc;
        const int64_t n = x.nc * x.c * x.batch;
        if (dense)
          absmax_dense<T>(p, n, amax, s);
        else
          launch_pdl(absmax_tensor_kernel<T>, dim3(grid_for(n / 8 + 1, 8)), dim3(kThreads), 0, s,
              p, x.c * x.batch, x.nc, x.s_c, vec_div(x.nc), amax);
      } else {
        for (int64_t b = 0; b < x.batch; ++b)
          launch_pdl(absmax_tensor_kernel<T>, dim3(grid_for(x.nc * x.c / 8 + 1, 8)), dim3(kThreads), 0, s,
              p + b * x.s_b, x.c, x.nc, x.s_c, vec_div(x.nc), amax);
      }
    } else {
      const int64_t col_blocks = (x.nc + 255) / 256;
      int64_t want_y = ((int64_t)sm_count() * 8 + col_blocks * x.batch - 1) / (col_blocks * x.batch);
      int64_t rows_per_block = (x.c + want_y - 1) / want_y;
      rows_per_block = (rows_per_block + 7) / 8 * 8;
      if (rows_per_block < 64) rows_per_block = 64;
      const int64_t gy = (x.c + rows_per_block - 1) / rows_per_block;
      dim3 grid((unsigned)col_blocks, (unsigned)gy, (unsigned)x.batch), block(32, 8);
      launch_pdl(absmax_cols_kernel<T>, dim3(grid), dim3(block), 0, s, p, x.nc, x.c, x.s_c, x.s_b, rows_per_block, amax);
    }
  }
  count_launch();
  QM_CUDA_OK(cudaGetLastError());
  return QM_OK;
}

// The shared-memory transposing kernels serve bf16 views whose contraction is strided and a multiple of 16
// long (codes and copy then go out in whole 16-byte vectors), in tiles of 128 contraction entries x 64 columns.
bool tile_transposable(const View& x) {
  return x.dtype == QM_DT_BF16 && !x.c_contig() && (x.c & 15) == 0 && (x.c + 127) / 128 <= 65535 && x.batch <= 65535;
}
bool tile_edges(const View& x) { return (x.c & 127) || (x.nc & 63); }
dim3 tile_grid(const View& x) { return dim3((unsigned)((x.nc + 63) / 64), (unsigned)((x.c + 127) / 128), (unsigned)x.batch); }
// Stochastic rounding takes them from two tiles for three SMs on: a thread draws 32 numbers in sequence there, 16 in the
// general kernel, which with fewer tiles is the faster one: 256 x 32 5.1 / 2.5 us, 1024 x 200 5.2 / 3.4, 512 x 1024 (64
// tiles) 3.8 / 3.4; 1024 x 1024 (128) 3.9 / 4.4, 4096 x 1024 9.0 / 10.8 (tile kernel / general kernel).
bool tile_form(const View& x, bool stochastic) {
  if (!tile_transposable(x)) return false;
  const dim3 g = tile_grid(x);
  return !stochastic || 3 * (int64_t)g.x * g.y * g.z >= 2 * (int64_t)sm_count();
}

template <typename T, int FMT>
qm_status quantize_t(const View& x, int gran, const float* delta, bool from_amax, float* delta_out,
                     uint32_t* err_word, uint8_t* codes, void* abs_copy, void* kmaj_copy, const Rounding& rnd,
                     cudaStream_t s) {
  const T* p = static_cast<const T*>(x.data);
  const int64_t ldc = qm_code_ld(x.c);
  DeltaSrc ds;
  ds.p = delta; ds.per_channel = gran == QM_GRAN_CHANNEL; ds.from_amax = from_amax ? 1 : 0;
  ds.qmax = fmt_qmax(FMT); ds.out = delta_out; ds.err_word = err_word;
  if (x.c_contig()) {
    const int64_t total = x.nc * x.batch * (ldc >> 4);
    if (total >= (1ll << 32) || x.nc >= (1ll << 32)) return QM_ERR_UNSUPPORTED;   // 32-bit chunk index
    const bool dense = x.dtype == QM_DT_BF16 && x.s_nc == x.c && (x.c & 15) == 0 && (x.batch == 1 || x.s_b == x.nc * x.c);
    if (dense && rnd.stochastic && !abs_copy) {
      launch_pdl(quantize_dense_sr_kernel<FMT>, dim3((unsigned)((total + kThreads - 1) / kThreads)), dim3(kThreads), 0, s,
                 reinterpret_cast<const uint4*>(x.data), (uint32_t)total, ds, FastDiv((uint32_t)(ldc >> 4)), (uint32_t)(ldc >> 4),
                 reinterpret_cast<uint4*>(codes), rnd);
    } else if (dense && !rnd.stochastic) {
      const uint4* src = reinterpret_cast<const uint4*>(x.data);
      const FastDiv by_chunks((uint32_t)(ldc >> 4));
      const bool big = total >= (int64_t)sm_count() * 8 * kThreads * 4;
      const bool wide = (reinterpret_cast<uintptr_t>(x.data) & 31) == 0;
      const int64_t per_block = (int64_t)kThreads * (big ? 4 : 1);
      const dim3 grid((unsigned)((total + per_block - 1) / per_block));
#define QM_QD(C, W)                                                                                                 \
  launch_pdl(quantize_dense_kernel<FMT, C, W>, grid, dim3(kThreads), 0, s, src, (uint32_t)total, ds, by_chunks, \
             (uint32_t)(ldc >> 4), reinterpret_cast<uint4*>(codes), reinterpret_cast<uint4*>(abs_copy))
      if (big) { if (wide) QM_QD(4, true); else QM_QD(4, false); }
      else { if (wide) QM_QD(1, true); else QM_QD(1, false); }
#undef QM_QD
    } else if (!ds.per_channel && !rnd.stochastic && !abs_copy) {
      MultiOut o{};
      o.codes[FMT] = codes; o.delta_out[FMT] = delta_out; o.err_word[FMT] = err_word;
      const dim3 grid((unsigned)((total + kThreads - 1) / kThreads));
      const FastDiv by_chunks((uint32_t)(ldc >> 4)), by_nc((uint32_t)x.nc);
      if (from_amax)
        launch_pdl(quantize_lines_kernel<T, 1 << FMT, false>, grid, dim3(kThreads), 0, s, p, (uint32_t)total, x.c, x.s_nc, x.s_b, by_chunks,
                   by_nc, reinterpret_cast<const uint32_t*>(delta), nullptr, o, ldc);
      else
        launch_pdl(quantize_lines_kernel<T, 1 << FMT, true>, grid, dim3(kThreads), 0, s, p, (uint32_t)total, x.c, x.s_nc, x.s_b, by_chunks,
                   by_nc, nullptr, delta, o, ldc);
    } else
    launch_pdl(quantize_rows_kernel<T, FMT>, dim3(grid_for(total, 16)), dim3(kThreads), 0, s, 
        p, x.nc, x.c, x.s_nc, x.batch, x.s_b, ds, FastDiv((uint32_t)(ldc >> 4)), FastDiv((uint32_t)x.nc),
        codes, ldc, static_cast<__nv_bfloat16*>(abs_copy), rnd);
    if (kmaj_copy) {
      // already contraction-major: a strided copy honours the parameter
      if (x.dtype != QM_DT_BF16) return QM_ERR_UNSUPPORTED;
      for (int64_t b = 0; b < x.batch; ++b)
        QM_CUDA_OK(cudaMemcpy2DAsync(static_cast<uint8_t*>(kmaj_copy) + b * x.nc * x.c * 2, x.c * 2,
                                     static_cast<const uint8_t*>(x.data) + b * x.s_b * 2, x.s_nc * 2,
                                     x.c * 2, x.nc, cudaMemcpyDeviceToDevice, s));
    }
  } else {
    if (!abs_copy && tile_form(x, rnd.stochastic)) {
#define QM_TT(KERNEL, ...)                                                                                      \
  launch_pdl(KERNEL, tile_grid(x), dim3(kThreads), 0, s, static_cast<const __nv_bfloat16*>(x.data), x.nc, x.c, x.s_c, x.s_b, ds, \
             codes, ldc, static_cast<__nv_bfloat16*>(kmaj_copy), ##__VA_ARGS__)
      if (!rnd.stochastic) {
        if (tile_edges(x)) QM_TT((quantize_transpose_tile_kernel<FMT, true>)); else QM_TT((quantize_transpose_tile_kernel<FMT, false>));
      } else {
        if (tile_edges(x)) QM_TT((quantize_transpose_tile_sr_kernel<FMT, true>), rnd);
        else QM_TT((quantize_transpose_tile_sr_kernel<FMT, false>), rnd);
      }
#undef QM_TT
      count_launch();
      QM_CUDA_OK(cudaGetLastError());
      return QM_OK;
    }
    if (!rnd.stochastic && x.dtype == QM_DT_BF16 && (x.c & 31) == 0 && (x.nc & 1) == 0 && (x.c + 255) / 256 <= 65535 &&
        ((x.nc + 63) / 64) * ((x.c + 255) / 256) * x.batch >= 4 * (int64_t)sm_count()) {
      dim3 grid((unsigned)((x.nc + 63) / 64), (unsigned)((x.c + 255) / 256), (unsigned)x.batch);
      launch_pdl(quantize_transpose_bf16_kernel<FMT>, dim3(grid), dim3(kThreads), 0, s, 
          static_cast<const __nv_bfloat16*>(x.data), x.nc, x.c, x.s_c, x.s_b, ds, codes, ldc,
          static_cast<__nv_bfloat16*>(abs_copy), static_cast<__nv_bfloat16*>(kmaj_copy));
      count_launch();
      QM_CUDA_OK(cudaGetLastError());
      return QM_OK;
    }
    dim3 grid((unsigned)((x.nc + 63) / 64), (unsigned)((ldc + 63) / 64), (unsigned)x.batch);
    launch_pdl(quantize_transpose_kernel<T, FMT>, dim3(grid), dim3(kThreads), 0, s, 
        p, x.nc, x.c, x.s_c, x.s_b, ds, codes, ldc, static_cast<__nv_bfloat16*>(abs_copy),
        static_cast<__nv_bfloat16*>(kmaj_copy), rnd);
  }
  count_launch();
  QM_CUDA_OK(cudaGetLastError());
  return QM_OK;
}

// Rows that the spread kernel takes: a multiple of 16 elements, so that codes have no padding, at most 8192 (two pieces for
// each thread of eight warps).  Short rows leave its lanes idle or, in bf16, have no more of them than one warp holds: those
// kernels are faster there, for one format.  Ragged rows and longer ones stay with the kernel that reads a row twice (one
// element at a time where it is ragged fp32), and a sharing of formats between rows of qm_quantize_formats is not built.
bool rows_spread(const View& x, int formats) {
  const int64_t least = formats > 1 ? 16 : x.dtype == QM_DT_BF16 ? 1040 : 272;
  return (x.c & 15) == 0 && x.c >= least && x.c <= 8192 && x.nc * x.batch < (1ll << 31) && x.nc < (1ll << 31);
}
template <typename T, int MASK>
qm_status rows_spread_t(const View& x, const MultiOut& o, cudaStream_t s) {
  const uint32_t rows = (uint32_t)(x.nc * x.batch);
  const int pieces = (int)(x.c / 16);
  const bool wide = ((reinterpret_cast<uintptr_t>(x.data) | (uintptr_t)(x.s_nc * sizeof(T)) | (x.batch > 1 ? (uintptr_t)(x.s_b * sizeof(T)) : 0)) & 31) == 0;
#define QM_SP(W, V)                                                                                                        \
  launch_pdl(scale_quantize_rows_spread_kernel<T, MASK, W, V>, dim3((unsigned)std::min<int64_t>((rows + 8 / W - 1) / (8 / W), 8ll * sm_count())), \
             dim3(kThreads), 0, s, static_cast<const T*>(x.data), rows, pieces, x.s_nc, x.s_b, FastDiv((uint32_t)x.nc), o, wide)
  if constexpr (sizeof(T) == 2) {
    if (pieces <= 64) QM_SP(1, 2);
    else if (pieces <= 128) QM_SP(2, 2);
    else if (pieces <= 256) QM_SP(4, 2);
    else QM_SP(8, 2);
  } else {
    if (pieces <= 32) QM_SP(1, 1);
    else if (pieces <= 64) QM_SP(2, 1);
    else if (pieces <= 128) QM_SP(4, 1);
    else if (pieces <= 256) QM_SP(8, 1);
    else QM_SP(8, 2);
  }
#undef QM_SP
  count_launch();
  QM_CUDA_OK(cudaGetLastError());
  return QM_OK;
}

template <typename T, int FMT>
qm_status scale_quantize_rows_t(const View& x, float* delta_out, uint8_t* codes, void* abs_copy,
                                uint32_t* err_word, cudaStream_t s) {
  const T* p = static_cast<const T*>(x.data);
  const int64_t rows = x.nc * x.batch, ldc = qm_code_ld(x.c), nvec = x.c / 8;
  const float qmax = fmt_qmax(FMT);
  if (!abs_copy && rows_spread(x, 1)) {
    MultiOut o{};
    o.codes[FMT] = codes; o.delta_out[FMT] = delta_out; o.err_word[FMT] = err_word;
    return rows_spread_t<T, 1 << FMT>(x, o, s);
  }
  if (x.dtype == QM_DT_BF16 && (x.c & 15) == 0 && x.c <= 4 * 256) {
    // the row fits in one warp's registers
    const unsigned blocks = (unsigned)((rows * 32 + kThreads - 1) / kThreads);
    const __nv_bfloat16* pb = static_cast<const __nv_bfloat16*>(x.data);
#define QM_SQR(V)                                                                                 \
  launch_pdl(scale_quantize_rows_reg_kernel<FMT, V>, dim3(blocks), dim3(kThreads), 0, s,                              \
      pb, x.nc, (int)nvec, x.s_nc, x.batch, x.s_b, qmax, delta_out, reinterpret_cast<uint2*>(codes), \
      reinterpret_cast<uint4*>(abs_copy), err_word)
    if (nvec <= 32) QM_SQR(1);
    else if (nvec <= 64) QM_SQR(2);
    else if (nvec <= 128) QM_SQR(4);
    else if (nvec <= 256) QM_SQR(8);
    else QM_SQR(16);
#undef QM_SQR
    count_launch();
    QM_CUDA_OK(cudaGetLastError());
    return QM_OK;
  }
#define QM_SQ(G)                                                                                   \
  launch_pdl(scale_quantize_rows_kernel<T, FMT, G>,                                                \
             dim3((unsigned)((rows * G + kThreads - 1) / kThreads)), dim3(kThreads), 0, s,         \
             p, x.nc, x.c, x.s_nc, x.batch, x.s_b, qmax, delta_out, codes, ldc,                    \
             static_cast<__nv_bfloat16*>(abs_copy), err_word)
  if (nvec <= 4) QM_SQ(4);
  else if (nvec <= 8) QM_SQ(8);
  else if (nvec <= 16) QM_SQ(16);
  else QM_SQ(32);
#undef QM_SQ
  count_launch();
  QM_CUDA_OK(cudaGetLastError());
  return QM_OK;
}

}  // namespace

qm_status launch_absmax(const View& x, int gran, uint32_t* amax_bits, cudaStream_t s) {
  return x.dtype == QM_DT_BF16 ? absmax_t<__nv_bfloat16>(x, gran, amax_bits, s)
                               : absmax_t<float>(x, gran, amax_bits, s);
}

// Which operands the two-launch form takes: fewer than 2^22 elements in both together, at most 2048 contiguous rows
// with a scale each, and no such rows with stochastic rounding, whose maxima nobody would have taken.  Whole probes, the
// general kernels / this form: 64 x 64 x 64 21.6 / 19.2 us, 1024 x 1024 x 1024 strided INT8 channel scales 36.7 / 31.7,
// 2048 x 1024 x 1024 33.9 / 31.7.  Beyond either line the operands' own kernels, lighter ones, fill the GPU: 16384 rows of 256 22.6 / 25.9;
// between 2^22 and 2^23 elements, 162 probes of all layouts, granularities and roundings, geometric mean 0.99 of the general kernels' speed, lowest 0.85
// (512 x 512 x 8000, one scale and a scale per row, 67.5 / 79.3; 3000 x 1000 x 2000 51.5 / 58.0; one operand rounded stochastically 61.2 / 65.7).  What gains there,
// both operands strided under channel scales (4096 x 1024 x 1024 42.4 / 38.9), loses at other shapes (100 x 50 x 30000 267 / 288, 8000 x 600 x 688 45.1 / 47.8).
static bool pair_size(const View& v) {
  return v.nc <= (1 << 22) && v.c <= (1 << 22) && v.batch <= (1 << 15) && v.nc * v.c <= (1ll << 22) && v.nc * v.c * v.batch <= (1ll << 22);
}
static bool pair_serves(const View& v, int gran, bool stochastic) {
  const bool rows = gran == QM_GRAN_CHANNEL && v.c_contig();
  return pair_size(v) && !(rows && (stochastic || v.nc * v.batch > 2048));
}

size_t pair_partial_words(const View& v, int gran) {
  if (!pair_size(v)) return 0;
  if (gran == QM_GRAN_TENSOR) return kPairBlocks;
  return v.c_contig() ? 0 : (size_t)(kPairSlices * v.nc * v.batch);
}

bool pair_prepare_serves(const View& l, int gran_l, bool draw_l, const View& r, int gran_r, bool draw_r) {
  return l.dtype == r.dtype && pair_serves(l, gran_l, draw_l) && pair_serves(r, gran_r, draw_r) &&
         (l.nc + r.nc) * l.c * l.batch < (1ll << 22);
}

qm_status launch_pair_prepare(const PairSide (&side)[2], uint32_t* control, uint32_t control_words, const uint32_t** flags, cudaStream_t s) {
  PairArgs a{};
  *flags = nullptr;
  a.control = control; a.control_words = control_words;
  for (int i = 0; i < 2; ++i) {
    const PairSide& in = side[i];
    PairOperand& o = a.op[i];
    o.v = in.v; o.fmt = in.fmt; o.per_channel = in.gran == QM_GRAN_CHANNEL;
    if (in.mn && !o.per_channel) {          // codes in storage order under one scale: those of the flipped view
      o.v.nc = in.v.c; o.v.c = in.v.nc; o.v.s_nc = in.v.s_c; o.v.s_c = in.v.s_nc;
    }
    const View& v = o.v;
    o.partial = in.partial; o.delta = in.delta; o.codes = in.codes;
    if (in.draw) { o.rnd.stochastic = 1; o.rnd.k0 = (uint32_t)in.draw->seed; o.rnd.k1 = (uint32_t)(in.draw->seed >> 32); o.rnd.stream = in.draw->stream; }
    const bool tiles = tile_form(v, in.draw != nullptr);
    const int64_t ldc = qm_code_ld(v.c);
    if (v.c_contig()) {
      const int64_t chunks = ldc >> 4, threads = v.nc * v.batch * (o.per_channel ? 32 : chunks);
      o.path = o.per_channel ? kPairRows : kPairChunks;
      o.blocks_quant = (int32_t)((threads + kThreads - 1) / kThreads);
      o.by_chunks = FastDiv((uint32_t)chunks); o.by_nc = FastDiv((uint32_t)v.nc);
    } else {
      o.path = in.mn ? kPairCols : tiles ? kPairTiles : kPairGeneral;
      o.col_lane_bits = col_lane_bits(v.nc);
      const int64_t cols = in.mn ? 8 << o.col_lane_bits : 64;
      o.gx = (uint32_t)((v.nc + cols - 1) / cols);
      o.gy = (uint32_t)(in.mn ? (v.c + kPairColRows - 1) / kPairColRows : tiles ? (v.c + 127) / 128 : (ldc + 63) / 64);
      o.by_gx = FastDiv(o.gx); o.by_gy = FastDiv(o.gy);
      o.blocks_quant = (int32_t)((int64_t)o.gx * o.gy * v.batch);
    }
    if (!o.per_channel) {
      const int64_t inner = v.c_contig() ? v.c : v.nc;
      o.lines = (uint32_t)(v.c_contig() ? v.nc : v.c);
      o.groups_per_line = (uint32_t)((inner + 7) / 8);
      o.total_groups = (uint32_t)(o.groups_per_line * (int64_t)o.lines * v.batch);
      o.by_groups = FastDiv(o.groups_per_line); o.by_lines = FastDiv(o.lines);
      const int64_t want = ((int64_t)o.total_groups + 4 * kThreads - 1) / (4 * kThreads);
      o.blocks_max = (int32_t)(want < kPairBlocks ? want : kPairBlocks);
      o.n_partial = o.blocks_max;
    } else if (!v.c_contig()) {
      // slices of at least 128 contraction entries
      const int64_t want = (v.c + 127) / 128;
      o.n_partial = (int32_t)(want < kPairSlices ? want : kPairSlices);
      o.max_cols = (uint32_t)((v.nc + 63) / 64);
      o.by_max_cols = FastDiv(o.max_cols);
      o.blocks_max = (int32_t)((int64_t)o.max_cols * v.batch * o.n_partial);
    }
  }
  const int f0 = side[0].fmt, f1 = side[1].fmt;
  const bool bf16 = side[0].v.dtype == QM_DT_BF16;
  for (int i = 0; i < 2; ++i) a.clusters[i] = once_clusters(a.op[i], bf16 ? 2 : 4);
  if (a.clusters[0] && a.clusters[1] && (a.clusters[0] + a.clusters[1]) * kOnceBlocks <= (uint32_t)kPrepareFlags) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((a.clusters[0] + a.clusters[1]) * kOnceBlocks); cfg.blockDim = dim3(kThreads); cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kOnceBlocks; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at; cfg.numAttrs = pdl_enabled() ? 2 : 1;
    const bool int8 = f0 == QM_FMT_INT8;                             // (INT8 goes with INT8 only)
    QM_CUDA_OK(cudaLaunchKernelEx(&cfg, bf16 ? (int8 ? pair_once_kernel<__nv_bfloat16, true> : pair_once_kernel<__nv_bfloat16, false>)
                                             : (int8 ? pair_once_kernel<float, true> : pair_once_kernel<float, false>), a));
    count_launch();
    *flags = control + kPrepareFlagWord;
    return QM_OK;
  }
  const unsigned maxima = (unsigned)(a.op[0].blocks_max + a.op[1].blocks_max);
  QM_CUDA_OK(launch_pdl(pair_max_kernel, dim3(maxima > 0 ? maxima : 1), dim3(kThreads), 0, s, a));
  const dim3 grid((unsigned)(a.op[0].blocks_quant + a.op[1].blocks_quant));
#define QM_PQ(F0, F1)                                                                                            \
  QM_CUDA_OK(bf16 ? launch_pdl(pair_quantize_kernel<__nv_bfloat16, F0, F1>, grid, dim3(kThreads), 0, s, a)        \
                  : launch_pdl(pair_quantize_kernel<float, F0, F1>, grid, dim3(kThreads), 0, s, a))
  if (f0 == QM_FMT_INT8) QM_PQ(QM_FMT_INT8, QM_FMT_INT8);          // (INT8 goes with INT8 only)
  else if (f0 == QM_FMT_E4M3 && f1 == QM_FMT_E4M3) QM_PQ(QM_FMT_E4M3, QM_FMT_E4M3);
  else if (f0 == QM_FMT_E4M3) QM_PQ(QM_FMT_E4M3, QM_FMT_E5M2);
  else if (f1 == QM_FMT_E4M3) QM_PQ(QM_FMT_E5M2, QM_FMT_E4M3);
  else QM_PQ(QM_FMT_E5M2, QM_FMT_E5M2);
#undef QM_PQ
  count_launch(2);
  return QM_OK;
}

bool many_serves(const View& x) {
  return x.dtype == QM_DT_BF16 && x.c_contig() && (x.c & 15) == 0 && (x.nc == 1 || x.s_nc == x.c) && (x.batch == 1 || x.s_b == x.nc * x.c) &&
         (reinterpret_cast<uintptr_t>(x.data) & 31) == 0 && x.nc * x.c * x.batch < (1ll << 35);
}

qm_status launch_prepare_many(const ManyTensor* t, int n, cudaStream_t s) {
  if (n < 1 || n > kManyTensors) return QM_ERR_INVALID_ARG;
  ManyList<ManyMax> m{};
  ManyList<ManyCodes> q{};
  m.n = q.n = n;
  int64_t total = 0;
  for (int i = 0; i < n; ++i) total += t[i].x.nc * t[i].x.c * t[i].x.batch / 16;
  // four chunks to a thread where that still gives an SM eight blocks
  const int chunks = total >= (int64_t)sm_count() * 8 * kThreads * 4 ? 4 : 1;
  uint32_t blocks_m = 0, blocks_q = 0;
  for (int i = 0; i < n; ++i) {
    const int64_t c = t[i].x.nc * t[i].x.c * t[i].x.batch / 16;                  // a chunk of 16 elements is a vector of 32 bytes
    m.e[i] = ManyMax{static_cast<const uint8_t*>(t[i].x.data), (uint64_t)c, t[i].amax, blocks_m};
    ManyCodes& e = q.e[i];
    e.x = static_cast<const uint8_t*>(t[i].x.data); e.amax = t[i].amax; e.chunks = (uint32_t)c; e.block0 = blocks_q;
    for (int f = 0; f < 3; ++f) { e.delta[f] = t[i].delta[f]; e.err[f] = t[i].err[f]; e.codes[f] = reinterpret_cast<uint4*>(t[i].codes[f]); }
    blocks_m += (uint32_t)((c + kThreads * kManyAhead - 1) / (kThreads * kManyAhead));
    blocks_q += (uint32_t)((c + kThreads * chunks - 1) / (kThreads * chunks));
  }
  QM_CUDA_OK(launch_pdl(absmax_many_kernel, dim3(blocks_m), dim3(kThreads), 0, s, m));
  QM_CUDA_OK(chunks == 4 ? launch_pdl(quantize_many_kernel<4>, dim3(blocks_q), dim3(kThreads), 0, s, q)
                         : launch_pdl(quantize_many_kernel<1>, dim3(blocks_q), dim3(kThreads), 0, s, q));
  count_launch(2);
  return QM_OK;
}

qm_status launch_share_amax(uint32_t* amax_bits, int64_t batch, int64_t groups, int64_t nc, cudaStream_t s) {
  const int64_t n = groups * nc;
  launch_pdl(share_amax_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, s, amax_bits, batch, groups, nc);
  count_launch();
  QM_CUDA_OK(cudaGetLastError());
  return QM_OK;
}

qm_status launch_finalize_delta(float* delta, int64_t n, int fmt, uint32_t* err_word, cudaStream_t s) {
  launch_pdl(finalize_delta_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, s, delta, n, fmt_qmax(fmt), err_word);
  count_launch();
  QM_CUDA_OK(cudaGetLastError());
  return QM_OK;
}

qm_status launch_quantize(const View& x, int fmt, int gran, const float* delta, bool from_amax,
                          float* delta_out, uint32_t* err_word, uint8_t* codes, void* abs_copy,
                          void* kmaj_copy, cudaStream_t s, const StochasticDraw* draw) {
  Rounding rnd{};
  if (draw) {
    rnd.stochastic = 1;
    rnd.k0 = (uint32_t)draw->seed; rnd.k1 = (uint32_t)(draw->seed >> 32); rnd.stream = draw->stream;
  }
#define QM_ARGS x, gran, delta, from_amax, delta_out, err_word, codes, abs_copy, kmaj_copy, rnd, s
#define QM_Q(T)                                                    \
  (fmt == QM_FMT_INT8   ? quantize_t<T, QM_FMT_INT8>(QM_ARGS)      \
   : fmt == QM_FMT_E4M3 ? quantize_t<T, QM_FMT_E4M3>(QM_ARGS)      \
                        : quantize_t<T, QM_FMT_E5M2>(QM_ARGS))
  return x.dtype == QM_DT_BF16 ? QM_Q(__nv_bfloat16) : QM_Q(float);
#undef QM_Q
#undef QM_ARGS
}

qm_status launch_quantize_multi(const View& x, int gran, const uint32_t* amax, int nf, const int* fmts,
                                float* const* delta_out, uint32_t* const* err_word, uint8_t* const* codes,
                                void* kmaj_copy, cudaStream_t s) {
  if (nf < 1 || nf > 3) return QM_ERR_INVALID_ARG;
  const int64_t ldc = qm_code_ld(x.c);
  int mask = 0;
  MultiOut o{};
  for (int k = 0; k < nf; ++k) {
    const int f = fmts[k];
    if (f < 0 || f > 2 || (mask & (1 << f))) return QM_ERR_INVALID_ARG;
    mask |= 1 << f;
    o.codes[f] = codes[k]; o.delta_out[f] = delta_out[k]; o.err_word[f] = err_word[k];
  }
  bool one_pass = nf > 1 && gran == QM_GRAN_TENSOR && (x.dtype == QM_DT_BF16 || x.c_contig());
  const int64_t total = x.nc * x.batch * (ldc >> 4);
  bool dense = false, transposing = false;
  if (one_pass && x.c_contig()) {
    dense = x.dtype == QM_DT_BF16 && x.s_nc == x.c && (x.c & 15) == 0 && (x.batch == 1 || x.s_b == x.nc * x.c);
    one_pass = total < (1ll << 32) && x.nc < (1ll << 32) && !kmaj_copy;
  } else if (one_pass) {
    transposing = tile_transposable(x);
    one_pass = transposing;
  }
  if (!one_pass) {
    // one launch per format; the first one also writes the contraction-major copy
    for (int k = 0; k < nf; ++k) {
      const qm_status st = launch_quantize(x, fmts[k], gran, reinterpret_cast<const float*>(amax), true, delta_out[k],
                                           err_word[k], codes[k], nullptr, k == 0 ? kmaj_copy : nullptr, s);
      if (st != QM_OK) return st;
    }
    return QM_OK;
  }
  if (dense) {
    const uint4* src = reinterpret_cast<const uint4*>(x.data);
    const bool big = total >= (int64_t)sm_count() * 8 * kThreads * 4;
    const int64_t per_block = (int64_t)kThreads * (big ? 4 : 1);
    const dim3 grid((unsigned)((total + per_block - 1) / per_block));
    const bool wide = (reinterpret_cast<uintptr_t>(x.data) & 31) == 0;
#define QM_DM(M)                                                                                                           \
  (big ? (wide ? launch_pdl(quantize_dense_multi_kernel<M, 4, true>, grid, dim3(kThreads), 0, s, src, (uint32_t)total, amax, o)    \
               : launch_pdl(quantize_dense_multi_kernel<M, 4, false>, grid, dim3(kThreads), 0, s, src, (uint32_t)total, amax, o))  \
       : (wide ? launch_pdl(quantize_dense_multi_kernel<M, 1, true>, grid, dim3(kThreads), 0, s, src, (uint32_t)total, amax, o)    \
               : launch_pdl(quantize_dense_multi_kernel<M, 1, false>, grid, dim3(kThreads), 0, s, src, (uint32_t)total, amax, o)))
    switch (mask) {
      case 3: QM_DM(3); break;
      case 5: QM_DM(5); break;
      case 6: QM_DM(6); break;
      default: QM_DM(7); break;
    }
#undef QM_DM
  } else if (!transposing) {
    const dim3 grid((unsigned)((total + kThreads - 1) / kThreads));
    const FastDiv by_chunks((uint32_t)(ldc >> 4)), by_nc((uint32_t)x.nc);
    const float* none = nullptr;
#define QM_LM(M)                                                                                                          \
  (x.dtype == QM_DT_BF16                                                                                                  \
       ? launch_pdl(quantize_lines_kernel<__nv_bfloat16, M, false>, grid, dim3(kThreads), 0, s, static_cast<const __nv_bfloat16*>(x.data), \
                    (uint32_t)total, x.c, x.s_nc, x.s_b, by_chunks, by_nc, amax, none, o, ldc)                            \
       : launch_pdl(quantize_lines_kernel<float, M, false>, grid, dim3(kThreads), 0, s, static_cast<const float*>(x.data), (uint32_t)total, \
                    x.c, x.s_nc, x.s_b, by_chunks, by_nc, amax, none, o, ldc))
    switch (mask) {
      case 3: QM_LM(3); break;
      case 5: QM_LM(5); break;
      case 6: QM_LM(6); break;
      default: QM_LM(7); break;
    }
#undef QM_LM
  } else {
    const __nv_bfloat16* src = static_cast<const __nv_bfloat16*>(x.data);
    __nv_bfloat16* km = static_cast<__nv_bfloat16*>(kmaj_copy);
#define QM_TM(M)                                                                                                                                          \
  launch_pdl(tile_edges(x) ? quantize_transpose_tile_multi_kernel<M, true> : quantize_transpose_tile_multi_kernel<M, false>, tile_grid(x), \
             dim3(kThreads), 0, s, src, x.nc, x.c, x.s_c, x.s_b, amax, o, ldc, km)
    switch (mask) {
      case 3: QM_TM(3); break;
      case 5: QM_TM(5); break;
      case 6: QM_TM(6); break;
      default: QM_TM(7); break;
    }
#undef QM_TM
  }
  count_launch();
  QM_CUDA_OK(cudaGetLastError());
  return QM_OK;
}

qm_status launch_quantize_cols(const View& x, const uint32_t* amax, int nf, const int* fmts, float* const* delta_out,
                               uint32_t* const* err_word, uint8_t* const* codes, cudaStream_t s) {
  if (x.dtype != QM_DT_BF16 || x.c_contig() || nf < 1 || nf > 3) return QM_ERR_INVALID_ARG;
  int mask = 0;
  MultiOut o{};
  for (int k = 0; k < nf; ++k) {
    const int f = fmts[k];
    if (f < 0 || f > 2 || (mask & (1 << f))) return QM_ERR_INVALID_ARG;
    mask |= 1 << f;
    o.codes[f] = codes[k]; o.delta_out[f] = delta_out[k]; o.err_word[f] = err_word[k];
  }
  // runs of rows that give every SM four blocks, of whole steps and at most 65535 of them
  const int lane_bits = col_lane_bits(x.nc);
  const int64_t col_blocks = (x.nc + (8 << lane_bits) - 1) / (8 << lane_bits), want = (4ll * sm_count() + col_blocks * x.batch - 1) / (col_blocks * x.batch);
  int64_t rows = (x.c + want - 1) / want;
  const int64_t step = 32 * (32 >> lane_bits);                          // four rows a thread
  rows = (rows + step - 1) / step * step;
  const dim3 grid((unsigned)col_blocks, (unsigned)((x.c + rows - 1) / rows), (unsigned)x.batch);
  if (col_blocks > 0x7fffffffll || x.batch > 65535) return QM_ERR_UNSUPPORTED;
  const __nv_bfloat16* p = static_cast<const __nv_bfloat16*>(x.data);
#define QM_QC(M) launch_pdl(quantize_cols_kernel<M>, grid, dim3(kThreads), 0, s, p, x.nc, x.c, x.s_c, x.s_b, rows, lane_bits, amax, o, qm_code_ld(x.nc))
  switch (mask) {
    case 1: QM_QC(1); break;
    case 2: QM_QC(2); break;
    case 3: QM_QC(3); break;
    case 4: QM_QC(4); break;
    case 5: QM_QC(5); break;
    case 6: QM_QC(6); break;
    default: QM_QC(7); break;
  }
#undef QM_QC
  count_launch();
  QM_CUDA_OK(cudaGetLastError());
  return QM_OK;
}

bool rows_from_one_read(const View& x) { return x.dtype == QM_DT_BF16 && rows_spread(x, 2); }

qm_status launch_scale_quantize_rows_multi(const View& x, int nf, const int* fmts, float* const* delta_out,
                                           uint32_t* const* err_word, uint8_t* const* codes, cudaStream_t s) {
  if (nf < 1 || nf > 3) return QM_ERR_INVALID_ARG;
  if (nf == 1 || !rows_from_one_read(x)) {
    for (int k = 0; k < nf; ++k) {
      const qm_status st = launch_scale_quantize_rows(x, fmts[k], delta_out[k], codes[k], nullptr, err_word[k], s);
      if (st != QM_OK) return st;
    }
    return QM_OK;
  }
  int mask = 0;
  MultiOut o{};
  for (int k = 0; k < nf; ++k) {
    const int f = fmts[k];
    if (f < 0 || f > 2 || (mask & (1 << f))) return QM_ERR_INVALID_ARG;
    mask |= 1 << f;
    o.codes[f] = codes[k]; o.delta_out[f] = delta_out[k]; o.err_word[f] = err_word[k];
  }
  switch (mask) {
    case 3: return rows_spread_t<__nv_bfloat16, 3>(x, o, s);
    case 5: return rows_spread_t<__nv_bfloat16, 5>(x, o, s);
    case 6: return rows_spread_t<__nv_bfloat16, 6>(x, o, s);
    default: return rows_spread_t<__nv_bfloat16, 7>(x, o, s);
  }
}

qm_status launch_scale_quantize_rows(const View& x, int fmt, float* delta_out, uint8_t* codes,
                                     void* abs_copy, uint32_t* err_word, cudaStream_t s) {
#define QM_Q(T)                                                                                       \
  (fmt == QM_FMT_INT8   ? scale_quantize_rows_t<T, QM_FMT_INT8>(x, delta_out, codes, abs_copy, err_word, s) \
   : fmt == QM_FMT_E4M3 ? scale_quantize_rows_t<T, QM_FMT_E4M3>(x, delta_out, codes, abs_copy, err_word, s) \
                        : scale_quantize_rows_t<T, QM_FMT_E5M2>(x, delta_out, codes, abs_copy, err_word, s))
  return x.dtype == QM_DT_BF16 ? QM_Q(__nv_bfloat16) : QM_Q(float);
#undef QM_Q
}

}  // namespace qm
