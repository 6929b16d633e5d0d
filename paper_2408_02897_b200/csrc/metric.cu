// Eq. 3 on materialised arrays, and the deterministic final reduction shared with the fused
// probe kernels.
#include <algorithm>

#include "qm_internal.h"
#include "reduce.cuh"

namespace qm {
namespace {

constexpr int kThreads = 256;

// where sum i (0 .. 3: BE, diff^2, C^2, D^2) and the maximum (4) lie in a record
__device__ __forceinline__ int record_field(int i) { return i == 0 ? 0 : i == 4 ? 1 : i + 1; }

// Eq. 3 sums of a short run of elements in fp32, folded into fp64 by the caller.
struct Run {
  float be = 0, mx = 0, d2 = 0, r2 = 0, n2 = 0;
  __device__ __forceinline__ void add(float c, float q, float d) {
    const float diff = c - q;
    const float b = d != 0.f ? __fdiv_rn(fabsf(diff), d) : 0.f;
    be += b; mx = fmaxf(mx, b);
    d2 = fmaf(diff, diff, d2); r2 = fmaf(c, c, r2); n2 = fmaf(d, d, n2);
  }
};

// Each block owns a contiguous slice (a multiple of four elements); the order of additions is fixed by the
// launch shape.  Bound by HBM: 12 bytes per element.  A thread has six 16-byte loads in flight
// (VEC: all three arrays start on 16 bytes): 151 MB in 59 us with 4-byte loads, 30 us so.
template <bool VEC>
__global__ void __launch_bounds__(kThreads)
metric_partials_kernel(const float* __restrict__ ref, const float* __restrict__ q,
                       const float* __restrict__ den, int64_t count, double* __restrict__ partials) {
  pdl_prologue();
  __shared__ double s[5][8];
  const int64_t per_block = ((count + gridDim.x - 1) / gridDim.x + 3) & ~(int64_t)3;
  const int64_t i0 = (int64_t)blockIdx.x * per_block;
  const int64_t i1 = min(count, i0 + per_block);
  double sbe = 0, sd2 = 0, sr2 = 0, sn2 = 0;
  float mbe = 0;
  // fp32 inside a run of eight, fp64 across runs
  auto fold = [&](const Run& f) { sbe += f.be; mbe = fmaxf(mbe, f.mx); sd2 += f.d2; sr2 += f.r2; sn2 += f.n2; };
  int64_t base = i0;
  if (VEC) {
    for (; base + kThreads * 8 <= i1; base += kThreads * 8) {
      const int64_t i = base + threadIdx.x * 4;
      float4 c[2], a[2], d[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        c[u] = __ldg(reinterpret_cast<const float4*>(ref + i + u * kThreads * 4));
        a[u] = __ldg(reinterpret_cast<const float4*>(q + i + u * kThreads * 4));
        d[u] = __ldg(reinterpret_cast<const float4*>(den + i + u * kThreads * 4));
      }
      Run f;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        f.add(c[u].x, a[u].x, d[u].x); f.add(c[u].y, a[u].y, d[u].y);
        f.add(c[u].z, a[u].z, d[u].z); f.add(c[u].w, a[u].w, d[u].w);
      }
      fold(f);
    }
  }
  for (; base < i1; base += kThreads * 8) {
    Run f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int64_t i = base + u * kThreads + threadIdx.x;
      if (i < i1) f.add(__ldg(ref + i), __ldg(q + i), __ldg(den + i));
    }
    fold(f);
  }
  const double v[4] = {sbe, sd2, sr2, sn2};
  const double x = block_record<4>(v, mbe, s);
  const int held = threadIdx.x >> 3;
  if ((threadIdx.x & 7) == 0 && held < 5) partials[(int64_t)blockIdx.x * kPartialDoubles + record_field(held)] = x;
}

// One block; thread t sums records t, t+256, ... in order, then a fixed order over lanes and warps.
__global__ void __launch_bounds__(kThreads)
metric_finalize_kernel(const double* __restrict__ partials, int n, uint64_t count,
                       const uint32_t* __restrict__ err_word, qm_metric_result* __restrict__ out) {
  pdl_prologue();
  __shared__ double s[5][8];
  __shared__ double tot[5];
  double v[4] = {0, 0, 0, 0};
  float mx = 0.f;
  for (int i = threadIdx.x; i < n; i += kThreads) {
    const double* p = partials + (int64_t)i * kPartialDoubles;
    v[0] += p[0]; mx = fmaxf(mx, (float)p[1]); v[1] += p[2]; v[2] += p[3]; v[3] += p[4];
  }
  const double x = block_record<4>(v, mx, s);
  const int held = threadIdx.x >> 3;
  if ((threadIdx.x & 7) == 0 && held < 5) tot[record_field(held)] = x;
  __syncthreads();
  if (threadIdx.x == 0) {                    // (the record may be in host memory: stores only, every field once)
    out->sum_be = tot[0]; out->max_be = tot[1]; out->sum_diff2 = tot[2];
    out->sum_ref2 = tot[3]; out->sum_den2 = tot[4];
    out->count = count;
    out->device_error = err_word ? *err_word : 0u;
    out->reserved = 0;
  }
}

}  // namespace

int metric_blocks(int64_t count) {
  int64_t want = (count + kThreads * 8 - 1) / (kThreads * 8);
  int64_t cap = (int64_t)sm_count() * 8;
  return (int)(want < 1 ? 1 : (want < cap ? want : cap));
}

qm_status launch_metric_partials(const float* ref, const float* q, const float* den, int64_t count,
                                 double* partials, int nblocks, cudaStream_t s) {
  const bool vec = ((reinterpret_cast<uintptr_t>(ref) | reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(den)) & 15) == 0;
  QM_CUDA_OK(launch_pdl(vec ? metric_partials_kernel<true> : metric_partials_kernel<false>, dim3((unsigned)nblocks), dim3(kThreads), 0, s,
                        ref, q, den, count, partials));
  count_launch();
  return QM_OK;
}

qm_status launch_metric_finalize(const double* partials, int n, uint64_t count,
                                 const uint32_t* err_word, qm_metric_result* out, cudaStream_t s) {
  QM_CUDA_OK(launch_pdl(metric_finalize_kernel, dim3(1), dim3(kThreads), 0, s, partials, n, count, err_word, out));
  count_launch();
  return QM_OK;
}

}  // namespace qm

// ---------------------------------------------------------------------------------------------
// qm_metric_noalloc: Eq. 3 reduction for callers that cannot allocate device memory.
//
// The per-block partial records of qm_metric normally live in a caller-provided workspace.  A
// caller that runs where cudaMalloc is off limits (a plug-in that is handed raw input/output
// pointers by its host application, code running inside a memory-pool-managed region, a
// latency-critical loop that must not touch the allocator) has nowhere to get that workspace
// from.  For them the library carries the scratch itself, as a fixed array in the module's
// device image: kNoAllocRecords partial records (40 KiB), present on every GPU that loads the
// library until the process ends.
namespace qm {
namespace {

constexpr int kNoAllocRecords = 1024;                         // 1024 x 5 doubles = 40 KiB
constexpr int64_t kNoAllocMaxCount = (int64_t)1 << 30;        // elements per input array

static __device__ __align__(256) double g_noalloc_partials[kNoAllocRecords * kPartialDoubles];

// In host code the array's name is only a handle for the runtime, not a device address: the
// address the kernels need is looked up once per device (with that device current) and cached.
double* g_noalloc_ptr[kMaxDevices] = {};

qm_status noalloc_scratch(double** out) {
  int dev = -1;
  QM_CUDA_OK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return QM_ERR_UNSUPPORTED;
  if (!g_noalloc_ptr[dev]) {
    double* p = nullptr;
    QM_CUDA_OK(cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_noalloc_partials));
    if (!p) return QM_ERR_CUDA;
    g_noalloc_ptr[dev] = p;
  }
  *out = g_noalloc_ptr[dev];
  return QM_OK;
}

}  // namespace
// ---- clearing the control words of several workspaces in one launch --------------------------
namespace {
__global__ void clear_many_kernel(const ClearList list) {
  pdl_prologue();
  const int w = blockIdx.x;                      // gridDim.y blocks per region
  uint32_t* p = static_cast<uint32_t*>(list.ptr[w]);
  const uint64_t n = list.words[w];
  for (uint64_t i = blockIdx.y * blockDim.x + threadIdx.x; i < n; i += gridDim.y * blockDim.x) p[i] = 0u;
}
}  // namespace

qm_status launch_clear_many(const ClearList& list, cudaStream_t s) {
  if (list.n < 1 || list.n > kClearMax) return QM_ERR_INVALID_ARG;
  // four words to a thread until the GPU has two blocks for each SM (2^20 maxima by eight blocks: 6.6 us of a scale call of 23.1)
  uint64_t most = 0;
  for (int i = 0; i < list.n; ++i) most = std::max(most, list.words[i]);
  const uint64_t cap = std::max(1, 2 * sm_count() / list.n), want = (most + 1023) / 1024;
  QM_CUDA_OK(launch_pdl(clear_many_kernel, dim3((unsigned)list.n, (unsigned)std::clamp<uint64_t>(want, 1, cap)), dim3(256), 0, s, list));
  count_launch();
  return QM_OK;
}

}  // namespace qm

extern "C" qm_status qm_metric_noalloc(const float* ref, const float* q, const float* den, int64_t count,
                                       qm_metric_result* out, void* stream) {
  using namespace qm;
  if (!ref || !q || !den || !out || count <= 0) return QM_ERR_INVALID_ARG;
  if (count > kNoAllocMaxCount) return QM_ERR_WORKSPACE_TOO_SMALL;   // beyond the built-in scratch's stated limit
  double* scratch = nullptr;
  qm_status st = noalloc_scratch(&scratch);
  if (st != QM_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int nb = metric_blocks(count);
  if (nb > kNoAllocRecords) nb = kNoAllocRecords;
  // Every record that the final reduction reads is overwritten by its block first, so nothing
  // in the shared array has to be cleared between calls.
  st = launch_metric_partials(ref, q, den, count, scratch, nb, s);
  if (st != QM_OK) return st;
  return launch_metric_finalize(scratch, nb, (uint64_t)count, nullptr, out, s);
}

extern "C" int64_t qm_metric_noalloc_max_count(void) { return qm::kNoAllocMaxCount; }
