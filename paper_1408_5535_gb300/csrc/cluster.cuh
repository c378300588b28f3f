// Device and launch helpers of the kernels that keep a whole small problem in one
// thread-block cluster (k_jdsmall.cu, k_expand.cu).
#pragma once
#include <cuda_runtime.h>

#include <atomic>

#include "common.cuh"
#include "kernels.h"

namespace ph {

// A row of Q values that another CTA may have written: from L2.
template <typename T, int Q>
__device__ __forceinline__ void ld_row(const T* p, T (&r)[Q]) {
  if constexpr (sizeof(T) * Q % 16 == 0) {
#pragma unroll
    for (int k = 0; k < Q; k += 16 / (int)sizeof(T)) {
      if constexpr (sizeof(T) == 8) {
        const double2 t = __ldcg(reinterpret_cast<const double2*>(p + k));
        r[k] = t.x;
        r[k + 1] = t.y;
      } else {
        const float4 t = __ldcg(reinterpret_cast<const float4*>(p + k));
        r[k] = t.x;
        r[k + 1] = t.y;
        r[k + 2] = t.z;
        r[k + 3] = t.w;
      }
    }
  } else {
#pragma unroll
    for (int k = 0; k < Q; ++k) r[k] = __ldcg(p + k);
  }
}

// out(row, :) = sum of val * X(col, :) over the entries of rows [r0, r1), L lanes
// per row, JT threads; row(i, acc) is called by one thread.  A row much longer than the
// mean would keep its lanes, and the cluster behind them, for len / L dependent gathers (one
// full row of 12,000 beside 6 entries per row: 2583 us per iteration of stage 1 for 185).
// Rows over ROW_LANE L entries wait for a whole warp, over ROW_WARP for the CTA: a rule of
// the length alone, so that sums repeat.
constexpr int ROW_LANE = 64, ROW_WARP = 4096;
constexpr int ROW_BIG = 512;   // more rows of ROW_WARP entries than the lines of the kernels let in
template <typename T, int Q>
__device__ __forceinline__ void spmm_add(const int* __restrict__ idx, const T* __restrict__ val, const T* X, int e,
                                         int e1, int step, T (&acc)[Q]) {
#pragma unroll 4
  for (; e < e1; e += step) {
    const int c = idx[e];
    const T a = val[e];
    T x[Q];
    ld_row<T, Q>(X + (size_t)c * Q, x);
#pragma unroll
    for (int k = 0; k < Q; ++k) acc[k] = fma(a, x[k], acc[k]);
  }
}
// (In line: a call, though never made, costs every step of an inner solve 0.5 us of 28.)
template <typename T, int Q, int JT, typename F>
__device__ __forceinline__ void spmm_long_rows(const int* __restrict__ ptr, const int* __restrict__ idx,
                                            const T* __restrict__ val, const T* X, int r0, int r1, int L, F row) {
  __shared__ int nbig, big[ROW_BIG];
  __shared__ T part[JT / 32][Q];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) nbig = 0;
  __syncthreads();
  T acc[Q];
  auto warp_row = [&](int i, int e, int step) {
#pragma unroll
    for (int k = 0; k < Q; ++k) acc[k] = T(0);
    spmm_add<T, Q>(idx, val, X, ptr[i] + e, ptr[i + 1], step, acc);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < Q; ++k) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
  };
  for (int base = r0 + 32 * warp; base < r1; base += JT) {
    const int mine = base + lane, len = mine < r1 ? ptr[mine + 1] - ptr[mine] : 0;
    for (unsigned todo = __ballot_sync(0xffffffffu, len > ROW_LANE * L); todo; todo &= todo - 1) {
      const int l = __ffs(todo) - 1, i = base + l;
      if (__shfl_sync(0xffffffffu, len, l) > ROW_WARP) {
        int at = lane == 0 ? atomicAdd(&nbig, 1) : 0;
        at = __shfl_sync(0xffffffffu, at, 0);
        if (at < ROW_BIG) {
          if (lane == 0) big[at] = i;
          continue;
        }
      }
      warp_row(i, lane, 32);
      if (lane == 0) row(i, acc);
    }
  }
  __syncthreads();
  for (int q = 0; q < min(nbig, ROW_BIG); ++q) {
    const int i = big[q];
    warp_row(i, tid, JT);
    if (lane == 0)
#pragma unroll
      for (int k = 0; k < Q; ++k) part[warp][k] = acc[k];
    __syncthreads();
    if (tid == 0) {
      for (int w = 1; w < JT / 32; ++w)
#pragma unroll
        for (int k = 0; k < Q; ++k) acc[k] += part[w][k];
      row(i, acc);
    }
    __syncthreads();
  }
}
// Whether rows [r0, r1) hold such a long one (for the whole CTA; a barrier).
template <int JT>
__device__ inline bool long_rows(const int* __restrict__ ptr, int r0, int r1, int L) {
  bool any = false;
  for (int i = r0 + threadIdx.x; i < r1; i += JT) any = any || ptr[i + 1] - ptr[i] > ROW_LANE * L;
  return __syncthreads_or(any);
}
template <typename T, int Q, int JT, typename F>
__device__ __forceinline__ void spmm_rows(const int* __restrict__ ptr, const int* __restrict__ idx,
                                          const T* __restrict__ val, const T* X, int r0, int r1, int L, bool any_long,
                                          F&& row) {
  const int per = JT / L, gl = threadIdx.x % L, gi = threadIdx.x / L;
  for (int base = r0; base < r1; base += per) {   // uniform trip count: the shuffles need whole warps
    const int i = base + gi;
    const int e0 = i < r1 ? ptr[i] : 0, e1 = i < r1 ? ptr[i + 1] : 0;
    const bool later = e1 - e0 > ROW_LANE * L;
    T acc[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) acc[k] = T(0);
    if (!later) spmm_add<T, Q>(idx, val, X, e0 + gl, e1, L, acc);
    for (int o = L / 2; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < Q; ++k) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
    if (i < r1 && gl == 0 && !later) row(i, acc);
  }
  if (any_long) spmm_long_rows<T, Q, JT>(ptr, idx, val, X, r0, r1, L, row);
}

// Lanes per row: as many as keep a row within a few rounds of gathers.
inline int cluster_lanes(double avg) { return avg <= 8.0 ? 1 : avg <= 32.0 ? 4 : 16; }

template <typename A>
inline cudaLaunchConfig_t cluster_config(A* at, int nc, int threads, size_t smem, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nc);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = nc;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

// CTAs of the kernel's cluster on this device: 16 where it can be placed with smem
// bytes, else 8, else 0 (the general form has to run).  Sets the kernel's attributes (up
// to smem_max bytes) at first use.
template <typename K>
int cluster_size(K kernel, int threads, size_t smem, size_t smem_max, std::atomic<int> (&known)[64]) {
  constexpr int NONE = -1;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  const int was = known[dev & 63].load(std::memory_order_acquire);
  if (was) return was == NONE ? 0 : was;
  if (cudaPeekAtLastError() != cudaSuccess) return 0;   // an earlier error is its caller's to see
  int nc = 0;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max) == cudaSuccess &&
      cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess)
    for (int c = 16; c >= 8 && nc == 0; c /= 2) {
      cudaLaunchAttribute at[1];
      const cudaLaunchConfig_t cfg = cluster_config(at, c, threads, smem, nullptr);
      int fit = 0;
      if (cudaOccupancyMaxActiveClusters(&fit, kernel, &cfg) == cudaSuccess && fit > 0) nc = c;
    }
  if (nc < 16) cudaGetLastError();
  known[dev & 63].store(nc ? nc : NONE, std::memory_order_release);
  return nc;
}

// False: the launch was refused, nothing runs.
template <typename K, typename G>
bool launch_cluster(K kernel, int nc, int threads, size_t smem, cudaStream_t s, const G& args) {
  cudaLaunchAttribute at[1];
  const cudaLaunchConfig_t cfg = cluster_config(at, nc, threads, smem, s);
  if (cudaLaunchKernelEx(&cfg, kernel, args) != cudaSuccess) {
    cudaGetLastError();                            // (an error that lasts is met again by the general form)
    return false;
  }
  count_launch();
  return true;
}

}  // namespace ph
