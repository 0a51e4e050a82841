// Deterministic reductions that end in the kernel that computes them: every block
// writes one partial per value, and the block that finishes last folds the
// partials in index order (no second launch).  The result does not depend on which
// block that is.
#pragma once
#include <cuda_runtime.h>

namespace nc {

template <bool MAX, typename T>
__device__ __forceinline__ T warp_fold(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const T w = __shfl_down_sync(0xffffffffu, v, o);
    v = MAX ? (v > w ? v : w) : v + w;
  }
  return v;
}

// Block sum (or maximum) of one value per thread, THREADS threads, valid in thread 0.
template <bool MAX, int THREADS, typename T>
__device__ __forceinline__ T block_fold(T v) {
  __shared__ T sh[THREADS / 32];
  v = warp_fold<MAX>(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();  // sh may still be read from a previous call
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  if (wid == 0) {
    v = lane < THREADS / 32 ? sh[lane] : T(0);
    v = warp_fold<MAX>(v);
  }
  return v;
}

// Block sums of N values per thread (the first cnt of them) to partial[q * gridDim.x +
// blockIdx.x].  FP32 folds by shuffles; in a block of more than eight warps, which may hold
// more than the WIDE_FROM elements of an ordinary one, the warps' sums meet in FP64, so that
// the sum keeps the bits that it has over several blocks.  An FP64 addition holds a
// scheduler's unit for 64 cycles whatever the number of active lanes, so FP64 values go
// through shared memory and one warp adds a value's eight warps before its five shuffle
// steps: 12 additions per value and block instead of 45.
// N <= 8.
template <int THREADS, typename T>
__device__ __forceinline__ T* block_buffer() {  // one for every N
  __shared__ T sh[sizeof(T) == 8 ? 8 * THREADS : 8 * (THREADS / 32)];
  return sh;
}
constexpr int WIDE_FROM = 2048;
template <int THREADS, int N, typename T>
__device__ __forceinline__ void block_values(const T (&v)[N], int cnt, double* partial) {
  static_assert(N <= 8, "the buffer holds 8 values");
  constexpr int W = THREADS / 32;
  T* const sh = block_buffer<THREADS, T>();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if constexpr (sizeof(T) == 8) {
    __syncthreads();  // sh may still be read from a previous call
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (q < cnt) sh[(q * W + wid) * 32 + lane] = v[q];
    __syncthreads();
    for (int q = wid; q < cnt; q += W) {
      T t = sh[q * W * 32 + lane];
#pragma unroll
      for (int w = 1; w < W; ++w) t += sh[(q * W + w) * 32 + lane];
      t = warp_fold<false>(t);
      if (lane == 0) partial[(long long)q * gridDim.x + blockIdx.x] = double(t);
    }
  } else {
    __syncthreads();
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (q < cnt) {
        const T t = warp_fold<false>(v[q]);
        if (lane == 0) sh[wid * 8 + q] = t;
      }
    __syncthreads();
    if constexpr (W <= 8) {
      if ((int)threadIdx.x < cnt) {
        T t = sh[threadIdx.x];
#pragma unroll
        for (int w = 1; w < W; ++w) t += sh[w * 8 + threadIdx.x];
        partial[(long long)threadIdx.x * gridDim.x + blockIdx.x] = double(t);
      }
    } else if ((int)(threadIdx.x & ~31u) < cnt * W) {  // W lanes a value
      const int q = threadIdx.x / W, w = threadIdx.x % W;
      double t = q < cnt ? double(sh[w * 8 + q]) : 0.0;
#pragma unroll
      for (int o = W / 2; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o, W);
      if (w == 0 && q < cnt) partial[(long long)q * gridDim.x + blockIdx.x] = t;
    }
  }
}

// Whether the calling block is the last of its grid to get here.  Its threads then
// see what every other block wrote before its own call.  The ticket, 0 on entry,
// is left at 0.
__device__ __forceinline__ bool last_block(unsigned* ticket) {
  __shared__ bool last;
  if (gridDim.x * gridDim.y * gridDim.z == 1) {  // no other block: no fence, no atomic
    __syncthreads();
    return true;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(ticket, 1u) == gridDim.x * gridDim.y * gridDim.z - 1;
    if (last) *ticket = 0;
  }
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// Sum (or maximum) of nb partials in a fixed order, valid in thread 0 (one block).
template <bool MAX, int THREADS>
__device__ __forceinline__ double fold_partials(int nb, const double* partial) {
  double v = 0.0;
  for (int b = threadIdx.x; b < nb; b += THREADS) {
    const double q = __ldcg(partial + b);
    v = MAX ? (v > q ? v : q) : v + q;
  }
  return block_fold<MAX, THREADS>(v);
}

// put(q, the sum of partial[q * nb ...]) for q < cnt, by one lane of the value's warp; a
// fixed order.
template <typename F>
__device__ __forceinline__ void fold_values(int cnt, int nb, const double* partial, F&& put) {
  const int lane = threadIdx.x & 31;
  for (int q = threadIdx.x >> 5; q < cnt; q += blockDim.x >> 5) {
    double v = 0.0;
    for (int b = lane; b < nb; b += 32) v += __ldcg(partial + (long long)q * nb + b);
    v = warp_fold<false>(v);
    if (lane == 0) put(q, v);
  }
}

// A smoother's squared norm and its reciprocal root.
__device__ __forceinline__ bool norm_ok(double s2) { return s2 > 0.0 && s2 < 1e300; }
__device__ __forceinline__ void put_norm(double* sig2, double* isig, double s2) {
  *sig2 = s2;
  *isig = norm_ok(s2) ? rsqrt(s2) : 0.0;
}
__device__ __forceinline__ double coef_over(double g, double s2) { return norm_ok(s2) ? g / s2 : 0.0; }

}  // namespace nc
