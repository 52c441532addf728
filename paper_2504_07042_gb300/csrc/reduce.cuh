// Deterministic block and grid reductions shared by the solver kernels.
// Every sum has a fixed order (a fixed grid, a fixed tree), so results do not
// depend on scheduling.  The grid-level sum is finished inside the producing
// kernel by the block that arrives last (a release fence and an atomic count).
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

namespace ax {
namespace red {

constexpr int kThreads = 256;  // block size of every kernel that uses these helpers

// Fixed-order block reduction of v into out[blockIdx.x] (double accumulation).
__device__ __forceinline__ void block_reduce_store(double v, double *out) {
  __shared__ double sh[kThreads / 32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  if (wid == 0) {
    v = lane < kThreads / 32 ? sh[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) *out = v;
  }
}

// Fixed-order block reduction of two values at once, out_a[blockIdx.x] and
// out_b[blockIdx.x], one CTA barrier.  Float: the warp-level tree stays on the
// FP32 pipe, the eight warp results are added in double.  Double: an addition
// costs a warp 64 cycles of its SM quarter's FP64 pipe whatever its lanes do,
// and a tree in every warp is 10 of them; through shared memory one warp adds
// up all of a's threads and another all of b's, 13 each for the whole block.
template <typename T>
__device__ __forceinline__ void block_reduce2_store(T a, T b, double *out_a, double *out_b) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if constexpr (sizeof(T) == 8) {
    __shared__ double sh[2][kThreads];
    sh[0][threadIdx.x] = a;
    sh[1][threadIdx.x] = b;
    __syncthreads();
    if (wid == 0 || (wid == 1 && out_b)) {
      double v = sh[wid][lane];
      for (int q = lane + 32; q < kThreads; q += 32) v += sh[wid][q];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
      if (lane == 0) *(wid == 0 ? out_a : out_b) = v;
    }
  } else {
    __shared__ double sh[2][kThreads / 32];
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_down_sync(0xffffffffu, a, o);
      b += __shfl_down_sync(0xffffffffu, b, o);
    }
    if (lane == 0) {
      sh[0][wid] = (double)a;
      sh[1][wid] = (double)b;
    }
    __syncthreads();
    if (wid == 0) {
      double va = lane < kThreads / 32 ? sh[0][lane] : 0.0, vb = lane < kThreads / 32 ? sh[1][lane] : 0.0;
      for (int o = kThreads / 64; o > 0; o >>= 1) {
        va += __shfl_down_sync(0xffffffffu, va, o);
        vb += __shfl_down_sync(0xffffffffu, vb, o);
      }
      if (lane == 0) {
        *out_a = va;
        if (out_b) *out_b = vb;
      }
    }
  }
}

// s[u] = the sum of node u's local copies, which lie together: c[u] of them at
// Y[b[u]] on (c = 0: nothing, s = 0), in order.  The copies of all U nodes are
// loaded together, one, one more (the copy across a face), then two at a time
// (edges, corners); an addition is issued only where some lane of the warp
// needs it: in float64 one that no lane needs would cost as much of GB300's
// FP64 pipe (2 per clock and SM) as one that all need.
template <typename T, int U, typename I>
__device__ __forceinline__ void gather_copies(const T *Y, const I b[U], const I c[U], T s[U]) {
  int top[U], most = 0;
#pragma unroll
  for (int u = 0; u < U; ++u) s[u] = c[u] > 0 ? __ldcg(Y + b[u]) : T(0);
#pragma unroll
  for (int u = 0; u < U; ++u) {
    top[u] = __reduce_max_sync(0xffffffffu, (int)c[u]);
    most = max(most, top[u]);
  }
  auto step = [&](int q0, auto cnt) {
    constexpr int n = decltype(cnt)::value;
    T v[U][n];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int q = 0; q < n; ++q) v[u][q] = q0 + q < c[u] ? __ldcg(Y + b[u] + q0 + q) : T(0);
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int q = 0; q < n; ++q)
        if (q0 + q < top[u]) s[u] += v[u][q];
  };
  if (most > 1) step(1, std::integral_constant<int, 1>{});
  for (int q0 = 2; q0 < most; q0 += 2) step(q0, std::integral_constant<int, 2>{});
}

// Returns true in the block that arrives last at *cnt (after every block has
// written its partial: a release fence before the count) and resets *cnt.
__device__ __forceinline__ bool arrive_last(unsigned *cnt) {
  __shared__ bool last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(cnt, 1u) == gridDim.x - 1;
    if (last) *cnt = 0u;
  }
  __syncthreads();
  return last;
}

// Fixed-order sum of partial[0..nb) by one block (the last to arrive), read
// past L1: the partials were written by other SMs in this launch.
__device__ __forceinline__ double sum_partials(const double *partial, int nb) {
  __shared__ double total;
  double s = 0.0;
  for (int q = threadIdx.x; q < nb; q += blockDim.x) s += __ldcg(partial + q);
  block_reduce_store(s, &total);
  __syncthreads();
  return total;
}

// Fixed-order sums of two partial arrays a[0..nb), b[0..nb) by one block
// (the last to arrive), read past L1.
__device__ __forceinline__ void sum_partials2(const double *pa, const double *pb, int nb, double &ta, double &tb) {
  __shared__ double total[2];
  double sa = 0.0, sb = 0.0;
  for (int q = threadIdx.x; q < nb; q += blockDim.x) {
    sa += __ldcg(pa + q);
    sb += __ldcg(pb + q);
  }
  block_reduce2_store<double>(sa, sb, &total[0], &total[1]);
  __syncthreads();
  ta = total[0];
  tb = total[1];
}

}  // namespace red
}  // namespace ax
