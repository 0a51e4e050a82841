// The FP32 smoother of a small level in one block.
//
// On a level of a few hundred elements a kernel does 1-3 us of work, and the chain of
// kernels of a smoothing (three per Arnoldi step) costs about 6 us each, launch and trips
// to L2 included.  Here one block keeps the whole smoothing in its shared memory: the
// basis, t = D^-1 v, the state, the diagonal and the element rows of the product, with
// __syncthreads() where the kernels ended.  A thread takes whole elements (elem_jvp_f2,
// elem_jtvp_f2) and then nodes.  One SM works on it, so it pays while the product takes
// less than the launches saved.  An FGMRES iteration of a mixed solve without / with it:
// 16^3 (levels 8^3 and 4^3 here) 790 / 657 us, 64^3 1998 / 1890; with 4^3 alone 700 and
// 1927.  6^3 (96^3): 3650 / 3588.  512 elements are what the shared memory holds: 222 KB
// at six steps.
//
// The arithmetic is that of smooth() in nc_solver.cu: the basis is unnormalised, dots
// and norms are summed in FP32 in a fixed order (over the warps in FP64 where the level has
// more unknowns than one block of the general kernels sums) and their quotients formed in FP64.
#include "nc_element_f2.cuh"
#include "nc_internal.cuh"
#include "nc_reduce.cuh"
#include "nc_smooth.cuh"

namespace nc {

namespace {

constexpr int BT = 256, BW = BT / 32;  // one element per thread and pass at 255 registers
constexpr int BK = 8;                  // largest number of smoothing steps
static_assert(BW == 8 && BK == 8, "k_smooth_block folds eight values of eight warps, eight lanes each");

struct BlockSmooth {
  LevelDev d;
  ElemConst<float> c;
  const float *x, *gam, *src, *diag, *b;
  float *z, *r;  // r: the residual b - A z as well, if not null
  int k, zero;
};

// Shared floats: k + 1 basis vectors, t, x and D, then 40 rows per element.
inline long long block_floats(const LevelDev& d, int k) { return (k + 4LL) * 5 * d.Nn + 40 * d.E; }

struct BlockScalars {
  double H[BK * (BK + 1)], sig2[BK + 1], isig[BK + 1], y[BK + 1], g[BK + 1];
  float warp[BW][BK], cf[BK], sc;
};
// What the dynamic part may take: 227 KB a block less the scalars.  The attribute that
// allows it belongs to the kernel, not to a context, and solves on other threads set it
// too, so every launch sets this value and not its own size.
constexpr int BLOCK_BYTES = 227 * 1024 - 1168;
static_assert(sizeof(BlockScalars) <= 1168, "the scalars fit what BLOCK_BYTES leaves");

template <bool TR>
__global__ void __launch_bounds__(BT, 1) k_smooth_block(const __grid_constant__ BlockSmooth a) {
  chained();
  const float* const b = fresh(a.b);
  float* const z = fresh(a.z);
  const float* const gam = fresh(a.gam);
  const float* const src = a.src ? fresh(a.src) : nullptr;
  extern __shared__ float sm[];
  __shared__ BlockScalars sh;
  auto& H = sh.H;
  double *const sig2 = sh.sig2, *const isig = sh.isig, *const y = sh.y, *const g = sh.g;
  auto& warp = sh.warp;
  float* const cf = sh.cf;
  float& sc = sh.sc;
  const int Nn = (int)a.d.Nn, N = 5 * Nn, E = (int)a.d.E, k = a.k;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int sx = a.d.nx + 1, sy = a.d.ny + 1;
  float *const V = sm, *const t = V + (k + 1) * N, *const xs = t + N, *const D = xs + N, *const Y = D + N;

  // Y <- the element rows of A t (directions zero at Dirichlet unknowns)
  auto rows = [&] {
    for (int e = tid; e < E; e += BT) {
      const int i = e % a.d.nx, m = e / a.d.nx, j = m % a.d.ny, l = m / a.d.ny;
      const int n0 = i + sx * (j + sy * l);
      float xe[5][8], ve[5][8], out[5][8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int n = n0 + (q & 1) + ((q >> 1) & 1) * sx + (q >> 2) * sx * sy;
        const uint8_t fl = a.d.flag[n];
#pragma unroll
        for (int f = 0; f < 5; ++f) {
          xe[f][q] = xs[f * Nn + n];
          ve[f][q] = (fl >> f) & 1 ? 0.0f : t[f * Nn + n];
        }
      }
      if (TR)
        elem_jtvp_f2(xe, ve, gam[e], src ? src[e] : 0.0f, a.c, out);
      else
        elem_jvp_f2(xe, ve, gam[e], src ? src[e] : 0.0f, a.c, out);
#pragma unroll
      for (int f = 0; f < 5; ++f)
#pragma unroll
        for (int q = 0; q < 8; ++q) Y[(8 * f + q) * E + e] = out[f][q];
    }
  };
  // (A t)_n from the rows; Dirichlet rows t_n
  auto gather = [&](int n, float w[5]) {
    const int i = n % sx, m = n / sx, j = m % sy, l = m / sy;
#pragma unroll
    for (int f = 0; f < 5; ++f) w[f] = 0.0f;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int ei = i - (q & 1), ej = j - ((q >> 1) & 1), el = l - (q >> 2);
      if (ei < 0 || ej < 0 || el < 0 || ei >= a.d.nx || ej >= a.d.ny || el >= a.d.nz) continue;
      const float* p = Y + ei + a.d.nx * (ej + a.d.ny * el);
#pragma unroll
      for (int f = 0; f < 5; ++f) w[f] += p[(8 * f + q) * E];
    }
    const uint8_t fl = a.d.flag[n];
#pragma unroll
    for (int f = 0; f < 5; ++f)
      if ((fl >> f) & 1) w[f] = t[f * Nn + n];
  };
  const bool wide = N > WIDE_FROM;
  // The warps' parts of value q, summed: by every lane, or with `wide` by eight lanes together
  // (lane & 7 the warp), valid in all of them.
  auto over_warps = [&](int q) -> double {
    if (!wide) {
      float v = 0.0f;
      for (int m = 0; m < BW; ++m) v += warp[m][q];
      return v;
    }
    double v = warp[lane & 7][q];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  // The squared norm of v_j from its per-thread parts, and its reciprocal root, which the
  // last warp forms while the others begin the next product.
  auto norm = [&](int j, float s) {
    s = warp_fold<false>(s);
    if (lane == 0) warp[wid][0] = s;
    __syncthreads();
    if (wid == BW - 1) {
      const double v2 = over_warps(0);
      if (lane == 0) put_norm(sig2 + j, isig + j, v2);
    }
  };

  for (int m = tid; m < N; m += BT) {
    xs[m] = fresh(a.x)[m];
    D[m] = fresh(a.diag)[m];
    if (!a.zero) t[m] = z[m];
  }
  __syncthreads();
  if (!a.zero) {
    rows();
    __syncthreads();
    for (int n = tid; n < Nn; n += BT) {
      float w[5];
      gather(n, w);
#pragma unroll
      for (int f = 0; f < 5; ++f) V[f * Nn + n] = b[f * Nn + n] - w[f];
    }
    __syncthreads();
  }
  float s = 0.0f;
  for (int m = tid; m < N; m += BT) {
    const float v = a.zero ? b[m] : V[m];
    V[m] = v;
    t[m] = v / D[m];
    s += v * v;
  }
  norm(0, s);
  for (int j = 0; j < k; ++j) {
    float* const w = V + (j + 1) * N;
    rows();
    __syncthreads();
    float dot[BK];
#pragma unroll
    for (int q = 0; q < BK; ++q) dot[q] = 0.0f;
    for (int n = tid; n < Nn; n += BT) {
      float u[5];
      gather(n, u);
#pragma unroll
      for (int f = 0; f < 5; ++f) w[f * Nn + n] = u[f];
#pragma unroll
      for (int q = 0; q < BK; ++q)
        if (q <= j) {
#pragma unroll
          for (int f = 0; f < 5; ++f) dot[q] = fmaf(V[q * N + f * Nn + n], u[f], dot[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < BK; ++q)
      if (q <= j) {
        const float v = warp_fold<false>(dot[q]);
        if (lane == 0) warp[wid][q] = v;
      }
    __syncthreads();
    if (tid < 8 * BW) {  // eight lanes a dot
      const int q = tid >> 3;
      const double v = over_warps(q);  // not used beyond j
      if ((tid & 7) == 0 && q <= j) {
        H[j * (k + 1) + q] = v;
        cf[q] = (float)(v * isig[q] * isig[q]);
      }
    } else if (tid == 8 * BW) {
      sc = (float)isig[j];
    }
    __syncthreads();
    s = 0.0f;
    for (int m = tid; m < N; m += BT) {
      float v = w[m];
#pragma unroll
      for (int q = 0; q < BK; ++q)
        if (q <= j) v -= cf[q] * V[q * N + m];
      v *= sc;
      w[m] = v;
      t[m] = v / D[m];
      s += v * v;
    }
    norm(j + 1, s);
  }
  __syncthreads();
  if (wid == 0) {
    warp_least_squares(k, H, k + 1, sig2, isig, y, g);
    if (lane < k) cf[lane] = (float)y[lane];
  }
  __syncthreads();
  for (int m = tid; m < N; m += BT) {
    float v = 0.0f;
#pragma unroll
    for (int q = 0; q < BK; ++q)
      if (q < k) v += cf[q] * V[q * N + m];
    v /= D[m];
    if (!a.zero) v += z[m];
    z[m] = v;
    t[m] = v;
  }
  if (a.r) {
    __syncthreads();
    rows();
    __syncthreads();
    for (int n = tid; n < Nn; n += BT) {
      float w[5];
      gather(n, w);
#pragma unroll
      for (int f = 0; f < 5; ++f) a.r[f * Nn + n] = b[f * Nn + n] - w[f];
    }
  }
}

}  // namespace

bool smooth_block(const LevelDev& d, const ElemConst<float>& c, const LevelBuf<float>& B, bool tr, int k, bool zero,
                  float* r, cudaStream_t s) {
  const long long bytes = 4 * block_floats(d, k);
  if (k > BK || d.E > SMOOTH_BLOCK_MAX || bytes > BLOCK_BYTES) return false;
  const auto kernel = tr ? k_smooth_block<true> : k_smooth_block<false>;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, BLOCK_BYTES) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  const BlockSmooth a{d, c, B.x, B.gam, B.src, B.diag, B.b, B.z, r, k, zero ? 1 : 0};
  launch(kernel, 1, BT, bytes, s, a);
  return true;
}

}  // namespace nc
