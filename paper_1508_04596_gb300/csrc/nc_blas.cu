// Vector kernels: casts, axpy variants, deterministic reductions and the fused
// Gram-Schmidt / Arnoldi passes of the Krylov solvers.
//
// Every kernel is HBM-bound: it walks its vectors in chunks of four elements,
// moved as 16-byte packets (float4- / 2 x double2-wide) when every pointer it
// touches is 16-byte aligned, and element by element otherwise; the n mod 4
// tail is taken by the first threads.  Multivectors are stored with a padded
// leading dimension (a multiple of 64 elements) so that every column is aligned.
//
// Reductions use a fixed partition that depends only on the vector length:
// each block folds a grid-stride range of chunks into one partial with a
// warp-shuffle tree, and the block that finishes last folds the partials in index
// order (nc_reduce.cuh; a second kernel for that cost 3.7 us per reduction, of 9.7 us
// in all on a vector of 10^5).  Results are bitwise reproducible from run to run.
#include <cstdint>
#include <type_traits>

#include "nc_internal.cuh"
#include "nc_reduce.cuh"
#include "nc_smooth.cuh"

namespace nc {

namespace {

constexpr int VT = 256;
constexpr int MAP_BLOCKS_MAX = 8 * 152;  // streaming kernels: one wave of 256-thread blocks

template <typename R>
struct __align__(16) P4 {
  R v[4];
};

inline bool al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

inline unsigned map_blocks(long long n) {
  long long b = (n / 4 + VT - 1) / VT;
  if (b < 1) b = 1;
  if (b > MAP_BLOCKS_MAX) b = MAP_BLOCKS_MAX;
  return (unsigned)b;
}

// One block up to 4,096 elements in FP64: four chunks a thread cost less than another block's
// fence, atomic and second read (2 us of the 4 a small reduction takes).  In FP32 a block
// sums no more than WIDE_FROM elements: its sum is FP32, those of blocks meet in FP64.
template <typename R>
inline int red_blocks(long long n) {
  const long long per = RED_THREADS * 8;
  static_assert(WIDE_FROM == RED_THREADS * 8, "an ordinary block's elements");
  long long b = sizeof(R) == 8 && n <= 2 * per ? 1 : (n + per - 1) / per;
  if (b < 1) b = 1;
  if (b > RED_BLOCKS_MAX) b = RED_BLOCKS_MAX;
  return (int)b;
}

template <typename R, bool VEC>
__device__ __forceinline__ void ld4(const R* __restrict__ p, long long c, R o[4]) {
  if (VEC) {
    const P4<R> t = reinterpret_cast<const P4<R>*>(p)[c];
#pragma unroll
    for (int u = 0; u < 4; ++u) o[u] = t.v[u];
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u) o[u] = p[4 * c + u];
  }
}

template <typename R, bool VEC>
__device__ __forceinline__ void st4(R* __restrict__ p, long long c, const R o[4]) {
  if (VEC) {
    P4<R> t;
#pragma unroll
    for (int u = 0; u < 4; ++u) t.v[u] = o[u];
    reinterpret_cast<P4<R>*>(p)[c] = t;
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u) p[4 * c + u] = o[u];
  }
}

// Chunk loop of a streaming kernel: chunks c < n/4 by grid stride (f4), then
// the tail element n4*4 + gid for gid < n mod 4 (f1).
template <typename F4, typename F1>
__device__ __forceinline__ void chunk_loop(long long n, F4&& f4, F1&& f1) {
  const long long n4 = n >> 2;
  const long long gid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long gs = (long long)gridDim.x * blockDim.x;
  for (long long c = gid; c < n4; c += gs) f4(c);
  if (gid < (n & 3)) f1(n4 * 4 + gid);
}

template <typename Rd, typename Rs, bool VEC>
__global__ void k_cast(long long n, const Rs* __restrict__ x, Rd* __restrict__ y) {
  chunk_loop(n, [&](long long c) {
    Rs a[4];
    Rd b[4];
    ld4<Rs, VEC>(x, c, a);
#pragma unroll
    for (int u = 0; u < 4; ++u) b[u] = Rd(a[u]);
    st4<Rd, VEC>(y, c, b);
  }, [&](long long i) { y[i] = Rd(x[i]); });
}

template <typename R, bool VEC>
__global__ void k_axpy(long long n, R a, const R* __restrict__ x, R* __restrict__ y) {
  chunk_loop(n, [&](long long c) {
    R xv[4], yv[4];
    ld4<R, VEC>(x, c, xv);
    ld4<R, VEC>(y, c, yv);
#pragma unroll
    for (int u = 0; u < 4; ++u) yv[u] += a * xv[u];
    st4<R, VEC>(y, c, yv);
  }, [&](long long i) { y[i] += a * x[i]; });
}

template <typename R, bool VEC>
__global__ void k_xpay(long long n, const R* __restrict__ x, R a, R* __restrict__ y) {
  chunk_loop(n, [&](long long c) {
    R xv[4], yv[4];
    ld4<R, VEC>(x, c, xv);
    ld4<R, VEC>(y, c, yv);
#pragma unroll
    for (int u = 0; u < 4; ++u) yv[u] = xv[u] + a * yv[u];
    st4<R, VEC>(y, c, yv);
  }, [&](long long i) { y[i] = x[i] + a * y[i]; });
}

template <typename R, bool VEC>
__global__ void k_waxpy(long long n, const R* __restrict__ x, R a, const R* __restrict__ y,
                        R* __restrict__ w) {
  chunk_loop(n, [&](long long c) {
    R xv[4], yv[4];
    ld4<R, VEC>(x, c, xv);
    ld4<R, VEC>(y, c, yv);
#pragma unroll
    for (int u = 0; u < 4; ++u) xv[u] += a * yv[u];
    st4<R, VEC>(w, c, xv);
  }, [&](long long i) { w[i] = x[i] + a * y[i]; });
}

template <typename R, bool VEC>
__global__ void k_scal(long long n, R a, R* __restrict__ y) {
  chunk_loop(n, [&](long long c) {
    R yv[4];
    ld4<R, VEC>(y, c, yv);
#pragma unroll
    for (int u = 0; u < 4; ++u) yv[u] *= a;
    st4<R, VEC>(y, c, yv);
  }, [&](long long i) { y[i] *= a; });
}

// a[u] -= sum_{q < k} cf[q] X_q[chunk c][u], four columns per round so that four
// packet loads per thread are in flight.
template <typename R, bool VEC>
__device__ __forceinline__ void sub_cols(const R* __restrict__ X, long long ld, int k, const R* cf,
                                         long long c, R a[4]) {
  int q = 0;
  for (; q + 4 <= k; q += 4) {
    R xv[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r) ld4<R, VEC>(X + (q + r) * ld, c, xv[r]);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] -= cf[q + r] * xv[r][u];
  }
  for (; q < k; ++q) {
    R xv[4];
    ld4<R, VEC>(X + q * ld, c, xv);
#pragma unroll
    for (int u = 0; u < 4; ++u) a[u] -= cf[q] * xv[u];
  }
}

// Block-level sum of one value per thread, result valid in thread 0.
template <typename T>
__device__ __forceinline__ T block_sum(T v) {
  return block_fold<false, RED_THREADS>(v);
}

// The last block's end of a reduction of cnt values (nc_reduce.cuh).
template <typename F>
__device__ __forceinline__ void finish(int cnt, const double* partial, unsigned* ticket, F&& put) {
  if (last_block(ticket)) fold_values(cnt, gridDim.x, partial, put);
}

// One pass of a multi-dot over y: NC columns from X on, and with SELF y . y.  All
// columns' packets of a chunk are loaded before any is used: with a test of the
// column count around each load one was in flight at a time (FP64, 10 columns of 10.7M:
// 315 us against 225 now and 176 at the FP64 pipe's rate; the whole Gram-Schmidt step
// 1063 -> 868 us, FP32 401 -> 369).  FP32 sums go to two accumulators per column.
template <typename R, bool VEC, int NC, bool SELF>
__device__ __forceinline__ void mdot_pass(long long n, const R* __restrict__ X, long long ld,
                                          const R* __restrict__ y, double* partial, double* partial_self) {
  constexpr int CH = 16 / sizeof(R), NA = sizeof(R) == 4 ? 2 : 1;
  struct __align__(16) Pk {
    R v[CH];
  };
  const long long nc = n / CH;
  const long long gid = blockIdx.x * (long long)RED_THREADS + threadIdx.x;
  const long long gs = (long long)gridDim.x * RED_THREADS;
  auto get = [&](const R* p, long long c, R o[CH]) {
    if (VEC) {
      const Pk t = reinterpret_cast<const Pk*>(p)[c];
#pragma unroll
      for (int u = 0; u < CH; ++u) o[u] = t.v[u];
    } else {
#pragma unroll
      for (int u = 0; u < CH; ++u) o[u] = p[CH * c + u];
    }
  };
  R acc[NC][NA], accs = R(0);
#pragma unroll
  for (int q = 0; q < NC; ++q)
#pragma unroll
    for (int t = 0; t < NA; ++t) acc[q][t] = R(0);
  for (long long c = gid; c < nc; c += gs) {
    R yv[CH], xv[NC][CH];
    get(y, c, yv);
#pragma unroll
    for (int q = 0; q < NC; ++q) get(X + q * ld, c, xv[q]);
#pragma unroll
    for (int u = 0; u < CH; ++u) {
      if (SELF) accs = fma(yv[u], yv[u], accs);
#pragma unroll
      for (int q = 0; q < NC; ++q) acc[q][u % NA] = fma(xv[q][u], yv[u], acc[q][u % NA]);
    }
  }
  if (gid < n - nc * CH) {
    const long long i = nc * CH + gid;
    const R yt = y[i];
    if (SELF) accs = fma(yt, yt, accs);
#pragma unroll
    for (int q = 0; q < NC; ++q) acc[q][0] = fma(X[q * ld + i], yt, acc[q][0]);
  }
  R v[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) v[q] = NA == 2 ? acc[q][0] + acc[q][NA - 1] : acc[q][0];
  block_values<RED_THREADS>(v, NC, partial);
  if (SELF) {
    const R w[1] = {accs};
    block_values<RED_THREADS>(w, 1, partial_self);
  }
}

// Columns of one pass over y: FP64 is bound by the FP64 pipe (one FMA per 8 bytes), FP32
// by HBM.
template <typename R> constexpr int mdot_cols() { return sizeof(R) == 8 ? 4 : 8; }

// out[i] = X_i . y for i < k, and with self out[k] = y . y (per-thread sums in R, partials
// in double), in passes of nearly equal numbers of columns; cf, if not null, gets
// out[i] / sig2[i]
template <typename R, bool VEC>
__global__ void __launch_bounds__(RED_THREADS, 4) k_mdot(long long n, int k, const R* __restrict__ X,
                                                         long long ld, const R* __restrict__ y, int self,
                                                         double* partial, double* out,
                                                         const double* sig2, double* cf,
                                                         unsigned* ticket) {
  constexpr int KB = mdot_cols<R>();
  const int passes = (k + KB - 1) / KB;
  double* const ps = partial + (long long)k * gridDim.x;
  if (k == 0) {
    R acc[1] = {R(0)};
    chunk_loop(n, [&](long long c) {
      R a[4];
      ld4<R, VEC>(y, c, a);
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[0] = fma(a[u], a[u], acc[0]);
    }, [&](long long i) { acc[0] = fma(y[i], y[i], acc[0]); });
    block_values<RED_THREADS>(acc, 1, ps);
  }
  for (int p = 0, i0 = 0; p < passes; ++p) {
    const int nc = (k - i0 + passes - p - 1) / (passes - p);
    const R* const Xp = X + i0 * ld;
    double* const pp = partial + (long long)i0 * gridDim.x;
    auto pass = [&](auto c) {
      constexpr int NC = decltype(c)::value;
      if constexpr (NC <= KB) {
        if (self && p == 0)
          mdot_pass<R, VEC, NC, true>(n, Xp, ld, y, pp, ps);
        else
          mdot_pass<R, VEC, NC, false>(n, Xp, ld, y, pp, nullptr);
      }
    };
    switch (nc) {
      case 1: pass(std::integral_constant<int, 1>()); break;
      case 2: pass(std::integral_constant<int, 2>()); break;
      case 3: pass(std::integral_constant<int, 3>()); break;
      case 4: pass(std::integral_constant<int, 4>()); break;
      case 5: pass(std::integral_constant<int, 5>()); break;
      case 6: pass(std::integral_constant<int, 6>()); break;
      case 7: pass(std::integral_constant<int, 7>()); break;
      default: pass(std::integral_constant<int, 8>());
    }
    i0 += nc;
  }
  finish(k + (self ? 1 : 0), partial, ticket, [&](int q, double v) {
    out[q] = v;
    if (cf) cf[q] = coef_over(v, sig2[q]);
  });
}

// One Arnoldi step of the smoother with an unnormalised basis, its k coefficients cf_i
// and the reciprocal norm of v_{k-1} in Hd (formed once, by the block that ended the
// dots, and not in every block: an FP64 division or root is a chain of a microsecond):
//   w <- (w - sum_i cf_i v_i) / ||v_{k-1}||,   t = w / D (if t),
// the squared norm of w and its reciprocal root into Hd; with ls the block that ends the
// norm also solves the smoother's least-squares problem (k <= LS_MAX).
constexpr int LS_MAX = 8;
template <typename R, bool VEC>
__global__ void __launch_bounds__(RED_THREADS) k_arnoldi_update(long long n, int k,
                                                                const R* __restrict__ X, long long ld,
                                                                const R* __restrict__ D,
                                                                R* __restrict__ w, R* __restrict__ t,
                                                                double* Hd, int ls, double* partial,
                                                                unsigned* ticket) {
  __shared__ R cf[MAX_RESTART + 1];
  __shared__ R sc_sh;
  for (int i = threadIdx.x; i < k; i += blockDim.x) cf[i] = R(Hd[HD_CF + i]);
  if (threadIdx.x == RED_THREADS - 1) sc_sh = R(Hd[HD_ISIG + k - 1]);
  __syncthreads();
  const R sc = sc_sh;
  R acc2 = R(0);
  chunk_loop(n, [&](long long c) {
    R a[4];
    ld4<R, VEC>(w, c, a);
    sub_cols<R, VEC>(X, ld, k, cf, c, a);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      a[u] *= sc;
      acc2 += a[u] * a[u];
    }
    st4<R, VEC>(w, c, a);
    if (t) {
      R dv[4];
      ld4<R, VEC>(D, c, dv);
#pragma unroll
      for (int u = 0; u < 4; ++u) dv[u] = a[u] / dv[u];
      st4<R, VEC>(t, c, dv);
    }
  }, [&](long long i) {
    R a = w[i];
    for (int q = 0; q < k; ++q) a -= cf[q] * X[q * ld + i];
    a *= sc;
    acc2 += a * a;
    w[i] = a;
    if (t) t[i] = a / D[i];
  });
  const R s = block_sum(acc2);
  if (threadIdx.x == 0) partial[blockIdx.x] = double(s);
  if (!last_block(ticket)) return;
  fold_values(1, gridDim.x, partial, [&](int, double v) { put_norm(Hd + HD_SIG2 + k, Hd + HD_ISIG + k, v); });
  if (ls) {
    __shared__ double H[LS_MAX * (LS_MAX + 1)], nrm[2][LS_MAX + 1], g[LS_MAX + 1];
    __syncthreads();
    for (int q = threadIdx.x; q < k * (k + 1); q += RED_THREADS)
      H[q] = __ldcg(Hd + (q / (k + 1)) * LDH + q % (k + 1));
    if ((int)threadIdx.x <= k) {
      nrm[0][threadIdx.x] = __ldcg(Hd + HD_SIG2 + threadIdx.x);
      nrm[1][threadIdx.x] = __ldcg(Hd + HD_ISIG + threadIdx.x);
    }
    __syncthreads();
    if (threadIdx.x < 32) warp_least_squares(k, H, k + 1, nrm[0], nrm[1], Hd + HD_Y, g);
  }
}

// First basis vector of the smoother: v0 = r (copied unless r is v0 itself),
// t = r / D, its norm into Hd.
template <typename R, bool VEC>
__global__ void __launch_bounds__(RED_THREADS) k_init_basis(long long n, const R* r,
                                                            const R* __restrict__ D, R* v0,
                                                            R* __restrict__ t, double* Hd,
                                                            double* partial, unsigned* ticket) {
  const bool copy = r != v0;
  R acc2 = R(0);
  chunk_loop(n, [&](long long c) {
    R a[4], dv[4];
    ld4<R, VEC>(r, c, a);
    ld4<R, VEC>(D, c, dv);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      acc2 += a[u] * a[u];
      dv[u] = a[u] / dv[u];
    }
    if (copy) st4<R, VEC>(v0, c, a);
    st4<R, VEC>(t, c, dv);
  }, [&](long long i) {
    const R a = r[i];
    acc2 += a * a;
    if (copy) v0[i] = a;
    t[i] = a / D[i];
  });
  const R s = block_sum(acc2);
  if (threadIdx.x == 0) partial[blockIdx.x] = double(s);
  finish(1, partial, ticket, [&](int, double v) { put_norm(Hd + HD_SIG2, Hd + HD_ISIG, v); });
}

// z (+)= (sum_i coef[i] X_i) / D   (no division when D is null)
template <typename R, bool VEC>
__global__ void k_combine(long long n, int k, const R* __restrict__ X, long long ld,
                          const double* __restrict__ coef, const R* __restrict__ D, R* z,
                          int accumulate) {
  __shared__ R cf[MAX_RESTART + 1];
  for (int i = threadIdx.x; i < k; i += blockDim.x) cf[i] = R(-coef[i]);
  __syncthreads();
  chunk_loop(n, [&](long long c) {
    R a[4] = {R(0), R(0), R(0), R(0)};
    sub_cols<R, VEC>(X, ld, k, cf, c, a);  // cf holds the negated coefficients
    if (D) {
      R dv[4];
      ld4<R, VEC>(D, c, dv);
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] /= dv[u];
    }
    if (accumulate) {
      R zv[4];
      ld4<R, VEC>(z, c, zv);
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] += zv[u];
    }
    st4<R, VEC>(z, c, a);
  }, [&](long long i) {
    R a = R(0);
    for (int q = 0; q < k; ++q) a -= cf[q] * X[q * ld + i];
    if (D) a /= D[i];
    z[i] = accumulate ? z[i] + a : a;
  });
}

// y -= sign * sum_i coef[i] X_i
template <typename R, bool VEC>
__global__ void k_maxpy(long long n, int k, const R* __restrict__ X, long long ld,
                        const double* __restrict__ coef, double sign, R* __restrict__ y) {
  __shared__ R cf[MAX_RESTART + 1];
  for (int i = threadIdx.x; i < k; i += blockDim.x) cf[i] = R(sign * coef[i]);
  __syncthreads();
  chunk_loop(n, [&](long long c) {
    R a[4];
    ld4<R, VEC>(y, c, a);
    sub_cols<R, VEC>(X, ld, k, cf, c, a);
    st4<R, VEC>(y, c, a);
  }, [&](long long i) {
    R a = y[i];
    for (int q = 0; q < k; ++q) a -= cf[q] * X[q * ld + i];
    y[i] = a;
  });
}

// y -= sign * sum_i coef[i] X_i with FP32 columns and an FP64 y (FP64 arithmetic,
// the same order of operations as k_maxpy<double> on the cast columns)
template <bool VEC>
__global__ void k_maxpy_f32x(long long n, int k, const float* __restrict__ X, long long ld,
                             const double* __restrict__ coef, double sign,
                             double* __restrict__ y) {
  __shared__ double cf[MAX_RESTART + 1];
  for (int i = threadIdx.x; i < k; i += blockDim.x) cf[i] = sign * coef[i];
  __syncthreads();
  chunk_loop(n, [&](long long c) {
    double a[4];
    ld4<double, VEC>(y, c, a);
    int q = 0;
    for (; q + 4 <= k; q += 4) {
      float xv[4][4];
#pragma unroll
      for (int r = 0; r < 4; ++r) ld4<float, VEC>(X + (q + r) * ld, c, xv[r]);
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int u = 0; u < 4; ++u) a[u] -= cf[q + r] * (double)xv[r][u];
    }
    for (; q < k; ++q) {
      float xv[4];
      ld4<float, VEC>(X + q * ld, c, xv);
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] -= cf[q] * (double)xv[u];
    }
    st4<double, VEC>(y, c, a);
  }, [&](long long i) {
    double a = y[i];
    for (int q = 0; q < k; ++q) a -= cf[q] * (double)X[q * ld + i];
    y[i] = a;
  });
}

// Second classical Gram-Schmidt pass with the normalisation folded in:
// y <- (y - sum_i h_i X_i) / nw,  nw = sqrt(q - sum_i h_i^2)  with q = ||y||^2 on
// entry (h and q from one fused multi-dot; X orthonormal, so nw is the norm of
// the corrected y).  nw is written to *nw_out; a vanishing nw leaves the
// vector unscaled (the caller sees nw = 0 and stops).
template <typename R, bool VEC>
__global__ void k_maxpy_scale(long long n, int k, const R* __restrict__ X, long long ld,
                              const double* __restrict__ h, const double* __restrict__ q,
                              double* nw_out, R* __restrict__ y) {
  __shared__ R cf[MAX_RESTART + 1];
  __shared__ R sc_sh;
  for (int i = threadIdx.x; i < k; i += blockDim.x) cf[i] = R(h[i]);
  if (threadIdx.x == 0) {  // FP64 scalar work once per block
    double hh = 0.0;
    for (int i = 0; i < k; ++i) hh += h[i] * h[i];
    const double nw2 = *q - hh;
    const double nw = nw2 > 0.0 ? sqrt(nw2) : 0.0;
    sc_sh = (nw > 0.0 && nw < 1e300) ? R(1.0 / nw) : R(1);
    if (blockIdx.x == 0) *nw_out = nw;
  }
  __syncthreads();
  const R sc = sc_sh;
  chunk_loop(n, [&](long long c) {
    R a[4];
    ld4<R, VEC>(y, c, a);
    sub_cols<R, VEC>(X, ld, k, cf, c, a);
#pragma unroll
    for (int u = 0; u < 4; ++u) a[u] *= sc;
    st4<R, VEC>(y, c, a);
  }, [&](long long i) {
    R a = y[i];
    for (int qq = 0; qq < k; ++qq) a -= cf[qq] * X[qq * ld + i];
    y[i] = a * sc;
  });
}

}  // namespace

// Packets need every pointer 16-byte aligned and, for a multivector, a leading
// dimension that keeps each column aligned.
template <typename R>
inline bool mv_aligned(const R* X, long long ld) {
  return al16(X) && ((ld * (long long)sizeof(R)) & 15) == 0;
}

template <typename Rd, typename Rs>
void vcast(long long n, const Rs* x, Rd* y, cudaStream_t s) {
  if (al16(x) && al16(y))
    k_cast<Rd, Rs, true><<<map_blocks(n), VT, 0, s>>>(n, x, y);
  else
    k_cast<Rd, Rs, false><<<map_blocks(n), VT, 0, s>>>(n, x, y);
}
template <typename R>
void vcopy(long long n, const R* x, R* y, cudaStream_t s) {
  cudaMemcpyAsync(y, x, sizeof(R) * n, cudaMemcpyDeviceToDevice, s);
}
template <typename R>
void vzero(long long n, R* x, cudaStream_t s) {
  cudaMemsetAsync(x, 0, sizeof(R) * n, s);
}
template <typename R>
void vaxpy(long long n, R a, const R* x, R* y, cudaStream_t s) {
  if (al16(x) && al16(y))
    k_axpy<R, true><<<map_blocks(n), VT, 0, s>>>(n, a, x, y);
  else
    k_axpy<R, false><<<map_blocks(n), VT, 0, s>>>(n, a, x, y);
}
template <typename R>
void vxpay(long long n, const R* x, R a, R* y, cudaStream_t s) {
  if (al16(x) && al16(y))
    k_xpay<R, true><<<map_blocks(n), VT, 0, s>>>(n, x, a, y);
  else
    k_xpay<R, false><<<map_blocks(n), VT, 0, s>>>(n, x, a, y);
}
template <typename R>
void vwaxpy(long long n, const R* x, R a, const R* y, R* w, cudaStream_t s) {
  if (al16(x) && al16(y) && al16(w))
    k_waxpy<R, true><<<map_blocks(n), VT, 0, s>>>(n, x, a, y, w);
  else
    k_waxpy<R, false><<<map_blocks(n), VT, 0, s>>>(n, x, a, y, w);
}
template <typename R>
void vscal(long long n, R a, R* y, cudaStream_t s) {
  if (al16(y))
    k_scal<R, true><<<map_blocks(n), VT, 0, s>>>(n, a, y);
  else
    k_scal<R, false><<<map_blocks(n), VT, 0, s>>>(n, a, y);
}
template <typename R>
static void mdot(long long n, int k, const R* X, long long ld, const R* y, int self, double* out,
                 const double* sig2, double* cf, double* partial, cudaStream_t s) {
  const int nb = red_blocks<R>(n);
  if ((k == 0 || mv_aligned(X, ld)) && al16(y))
    k_mdot<R, true><<<nb, RED_THREADS, 0, s>>>(n, k, X, ld, y, self, partial, out, sig2, cf,
                                               red_ticket(partial));
  else
    k_mdot<R, false><<<nb, RED_THREADS, 0, s>>>(n, k, X, ld, y, self, partial, out, sig2, cf,
                                                red_ticket(partial));
}
template <typename R>
void vmdot(long long n, int k, const R* X, long long ld, const R* y, double* out, double* partial,
           cudaStream_t s) {
  mdot(n, k, X, ld, y, 0, out, nullptr, nullptr, partial, s);
}
template <typename R>
void vmdot_self(long long n, int k, const R* X, long long ld, const R* y, double* out,
                double* partial, cudaStream_t s) {
  mdot(n, k, X, ld, y, 1, out, nullptr, nullptr, partial, s);
}
template <typename R>
void vmdot_cf(long long n, int k, const R* X, long long ld, const R* y, double* out, const double* sig2,
              double* cf, double* partial, cudaStream_t s) {
  mdot(n, k, X, ld, y, 0, out, sig2, cf, partial, s);
}
template <typename R>
void vinit_basis(long long n, const R* r, const R* D, R* v0, R* t, double* Hd, double* partial,
                 cudaStream_t s) {
  const int nb = red_blocks<R>(n);
  if (al16(r) && al16(D) && al16(v0) && al16(t))
    k_init_basis<R, true><<<nb, RED_THREADS, 0, s>>>(n, r, D, v0, t, Hd, partial, red_ticket(partial));
  else
    k_init_basis<R, false><<<nb, RED_THREADS, 0, s>>>(n, r, D, v0, t, Hd, partial, red_ticket(partial));
}
template <typename R>
void varnoldi_update(long long n, int k, const R* X, long long ld, const R* D, R* w, R* t, double* Hd,
                     bool ls, double* partial, cudaStream_t s) {
  const int nb = red_blocks<R>(n), fused = ls && k <= LS_MAX;
  if (mv_aligned(X, ld) && al16(D) && al16(w) && al16(t))
    k_arnoldi_update<R, true><<<nb, RED_THREADS, 0, s>>>(n, k, X, ld, D, w, t, Hd, fused, partial,
                                                         red_ticket(partial));
  else
    k_arnoldi_update<R, false><<<nb, RED_THREADS, 0, s>>>(n, k, X, ld, D, w, t, Hd, fused, partial,
                                                          red_ticket(partial));
  if (ls && !fused) small_ls(Hd, k, s);
}
template <typename R>
void vcombine(long long n, int k, const R* X, long long ld, const double* coef, const R* D, R* z,
              bool accumulate, cudaStream_t s) {
  if (mv_aligned(X, ld) && al16(D) && al16(z))
    k_combine<R, true><<<map_blocks(n), VT, 0, s>>>(n, k, X, ld, coef, D, z, accumulate ? 1 : 0);
  else
    k_combine<R, false><<<map_blocks(n), VT, 0, s>>>(n, k, X, ld, coef, D, z, accumulate ? 1 : 0);
}
template <typename R>
void vmaxpy(long long n, int k, const R* X, long long ld, const double* coef, double sign, R* y,
            cudaStream_t s) {
  if (mv_aligned(X, ld) && al16(y))
    k_maxpy<R, true><<<map_blocks(n), VT, 0, s>>>(n, k, X, ld, coef, sign, y);
  else
    k_maxpy<R, false><<<map_blocks(n), VT, 0, s>>>(n, k, X, ld, coef, sign, y);
}
template <typename R>
void vmaxpy_scale(long long n, int k, const R* X, long long ld, const double* h, const double* q,
                  double* nw_out, R* y, cudaStream_t s) {
  if (mv_aligned(X, ld) && al16(y))
    k_maxpy_scale<R, true><<<map_blocks(n), VT, 0, s>>>(n, k, X, ld, h, q, nw_out, y);
  else
    k_maxpy_scale<R, false><<<map_blocks(n), VT, 0, s>>>(n, k, X, ld, h, q, nw_out, y);
}
void vmaxpy_f32x(long long n, int k, const float* X, long long ld, const double* coef,
                 double sign, double* y, cudaStream_t s) {
  if (mv_aligned(X, ld) && al16(y))
    k_maxpy_f32x<true><<<map_blocks(n), VT, 0, s>>>(n, k, X, ld, coef, sign, y);
  else
    k_maxpy_f32x<false><<<map_blocks(n), VT, 0, s>>>(n, k, X, ld, coef, sign, y);
}
template void vcast<float, double>(long long, const double*, float*, cudaStream_t);
template void vcast<double, float>(long long, const float*, double*, cudaStream_t);
#define NC_INST(R)                                                                             \
  template void vcopy<R>(long long, const R*, R*, cudaStream_t);                               \
  template void vzero<R>(long long, R*, cudaStream_t);                                         \
  template void vaxpy<R>(long long, R, const R*, R*, cudaStream_t);                            \
  template void vxpay<R>(long long, const R*, R, R*, cudaStream_t);                            \
  template void vwaxpy<R>(long long, const R*, R, const R*, R*, cudaStream_t);                 \
  template void vscal<R>(long long, R, R*, cudaStream_t);                                      \
  template void vmdot<R>(long long, int, const R*, long long, const R*, double*, double*,      \
                         cudaStream_t);                                                        \
  template void vmdot_self<R>(long long, int, const R*, long long, const R*, double*, double*, \
                              cudaStream_t);                                                   \
  template void vmdot_cf<R>(long long, int, const R*, long long, const R*, double*,            \
                            const double*, double*, double*, cudaStream_t);                    \
  template void vinit_basis<R>(long long, const R*, const R*, R*, R*, double*, double*,        \
                               cudaStream_t);                                                  \
  template void varnoldi_update<R>(long long, int, const R*, long long, const R*, R*, R*,      \
                                   double*, bool, double*, cudaStream_t);                      \
  template void vcombine<R>(long long, int, const R*, long long, const double*, const R*, R*,  \
                            bool, cudaStream_t);                                               \
  template void vmaxpy<R>(long long, int, const R*, long long, const double*, double, R*,      \
                          cudaStream_t);                                                       \
  template void vmaxpy_scale<R>(long long, int, const R*, long long, const double*,            \
                                const double*, double*, R*, cudaStream_t);
NC_INST(double)
NC_INST(float)
#undef NC_INST

}  // namespace nc
