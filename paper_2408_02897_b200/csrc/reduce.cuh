// Sums of several values over a block of 256 threads, for records that are written once per block: what such a record costs is
// a chain of dependent exchanges, so values are spread over the lanes while they are added (nine values: 12 exchanges
// of doubles instead of 45) and the warps' sums are added side by side.  The order of additions is fixed.
#pragma once
#include <cstdint>

namespace qm {
namespace {

// Adds v[0 .. N-1] over the warp.  On return `index` (0 on entry) says which sum this lane holds, `left` (N on entry) is not
// positive in lanes that hold none, and the lanes that differ in the bits below the returned-by-reference `below` hold the same one.
template <int N>
__device__ __forceinline__ double warp_sums(const double (&v)[N], int lane, int o, int& index, int& left, int& below) {
  if constexpr (N == 1) {
    double x = v[0];
    below = 2 * o;
#pragma unroll
    for (; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
  } else {
    constexpr int H = (N + 1) / 2;
    const bool up = lane & o;
    double a[H];
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const double lo = v[i], hi = i + H < N ? v[i + H] : 0.0;
      a[i] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, o);
    }
    index += up ? H : 0;
    left = up ? left - H : (left < H ? left : H);
    return warp_sums<H>(a, lane, o >> 1, index, left, below);
  }
}

// N sums and a maximum (of floats that are neither negative nor NaN) over the block's 256 threads; thread 8 i + k returns sum i
// for i < N, the maximum for i = N.  All threads call; red may be reused after a barrier.
template <int N>
__device__ __forceinline__ double block_record(const double (&v)[N], float mx, double (&red)[N + 1][8], int t = threadIdx.x) {
  const int lane = t & 31, warp = t >> 5;
  int index = 0, left = N, below;
  const double x = warp_sums<N>(v, lane, 16, index, left, below);
  const uint32_t m = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
  if (left > 0 && (lane & (below - 1)) == 0) red[index][warp] = x;
  if (lane == 0) red[N][warp] = (double)__uint_as_float(m);
  __syncthreads();
  double y = 0.0;
  if (t < ((8 * (N + 1) + 31) & ~31)) {                    // whole warps
    const int i = t >> 3;
    if (i <= N) y = red[i][t & 7];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      const double z = __shfl_xor_sync(0xffffffffu, y, o);
      y = i == N ? fmax(y, z) : y + z;
    }
  }
  return y;
}

}  // namespace
}  // namespace qm
