// Direct solve on the coarsest multigrid level.
//
// The coarsest grid is small (e.g. 2^3 or 3^3 elements, a few hundred unknowns),
// so instead of many Krylov iterations -- each a dozen kernel launches on a
// handful of elements -- its Jacobian is formed explicitly and inverted once
// per linearisation:
//   1. a kernel computes every column of every element Jacobian J_e in FP64
//      (the element tangent with unit directions; Dirichlet columns are zero),
//   2. the host assembles the dense matrix (Dirichlet rows identity, Dirichlet
//      columns removed from interior rows, the same operator as nc_jvp); it is
//      inverted by Gauss-Jordan elimination with partial pivoting in FP64, on the host
//      for the smallest systems, else on the device,
//   3. the inverse (in the cycle's precision) is applied with one dense
//      matrix-vector kernel: one warp per row, fixed-order shuffle reduction; the
//      transpose is stored after it, so that the adjoint's cycle reads rows too (a
//      thread per column took 39 us at 320 unknowns, 3.3 us by rows).
#include <cmath>
#include <cstring>
#include <vector>

#include "nc_internal.cuh"

namespace nc {
nc_status set_err(nc_ctx* ctx, nc_status st, const std::string& msg);
nc_status cuda_check(nc_ctx* ctx, cudaError_t e, const char* what);
}  // namespace nc

namespace nc {

namespace {

// One block per element, one thread per column k = f*8 + a of J_e.
template <typename R>
__global__ void k_coarse_elem_jac(LevelDev d, ElemConst<double> c, const R* __restrict__ x,
                                  const R* __restrict__ gam, const R* __restrict__ src,
                                  double* Jel) {
  const long long e = blockIdx.x;
  const int k = threadIdx.x;
  if (k >= 40 || e >= d.E) return;
  int i, j, kk;
  elem_ijk(d, e, i, j, kk);
  const long long sy = d.nx + 1, sz = (long long)(d.nx + 1) * (d.ny + 1);
  const long long n0 = i + sy * (j + (long long)(d.ny + 1) * kk);
  double xe[5][8], ve[5][8], out[5][8];
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const long long n = n0 + (a & 1) + ((a >> 1) & 1) * sy + ((a >> 2) & 1) * sz;
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      xe[f][a] = (double)x[f * d.Nn + n];
      ve[f][a] = 0.0;
    }
  }
  const int fk = k / 8, ak = k % 8;
  const long long nk = n0 + (ak & 1) + ((ak >> 1) & 1) * sy + ((ak >> 2) & 1) * sz;
  double* col = Jel + (e * 40 + k) * 40;
  if ((d.flag[nk] >> fk) & 1) {  // Dirichlet column: removed
    for (int r = 0; r < 40; ++r) col[r] = 0.0;
    return;
  }
  ve[fk][ak] = 1.0;
  elem_jvp<double>(xe, ve, (double)gam[e], src ? (double)src[e] : 0.0, c, out);
#pragma unroll
  for (int g = 0; g < 5; ++g)
#pragma unroll
    for (int b = 0; b < 8; ++b) col[g * 8 + b] = out[g][b];
}

// z = A b: one warp per row.
template <typename R>
__global__ void k_dense_gemv(int n, const R* __restrict__ A, const R* __restrict__ b,
                             R* __restrict__ z) {
  const int row = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= n) return;
  const R* a = A + (size_t)row * n;
  R acc = R(0);
  for (int j = lane; j < n; j += 32) acc += a[j] * b[j];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if (lane == 0) z[row] = acc;
}

// In-place Gauss-Jordan inverse with partial pivoting (row-major n x n).
// Returns false if a pivot vanishes (the coarse operator is singular).
bool gauss_jordan_inverse(std::vector<double>& A, int n) {
  std::vector<int> perm(n);
  for (int p = 0; p < n; ++p) {
    int q = p;
    double best = std::fabs(A[(size_t)p * n + p]);
    for (int i = p + 1; i < n; ++i) {
      const double v = std::fabs(A[(size_t)i * n + p]);
      if (v > best) { best = v; q = i; }
    }
    perm[p] = q;
    if (!(best > 0.0) || !std::isfinite(best)) return false;
    if (q != p)
      for (int j = 0; j < n; ++j) std::swap(A[(size_t)p * n + j], A[(size_t)q * n + j]);
    double* rp = &A[(size_t)p * n];
    const double inv = 1.0 / rp[p];
    rp[p] = 1.0;
    for (int j = 0; j < n; ++j) rp[j] *= inv;
    for (int i = 0; i < n; ++i) {
      if (i == p) continue;
      double* ri = &A[(size_t)i * n];
      const double f = ri[p];
      if (f == 0.0) continue;
      ri[p] = 0.0;
      for (int j = 0; j < n; ++j) ri[j] -= f * rp[j];
    }
  }
  // undo the row interchanges as column interchanges, in reverse order
  for (int p = n - 1; p >= 0; --p) {
    const int q = perm[p];
    if (q != p)
      for (int i = 0; i < n; ++i) std::swap(A[(size_t)i * n + p], A[(size_t)i * n + q]);
  }
  return true;
}

// ---- the same elimination on the device
// The largest candidate for a pivot among a block's rows, with its sign.
struct GjCand {
  double v;
  int row, pad;
};
constexpr int GJ_W = 8;  // rows per block, a warp each

// Whether candidate (v, row) goes before (w, row2): larger in size, ties to the first row.
__device__ __forceinline__ bool gj_before(double v, int row, double w, int row2) {
  return fabs(v) > fabs(w) || (fabs(v) == fabs(w) && row < row2);
}

// Step p: in -> out (n x n each, n <= 32 NV), a launch per step, a warp per row.  cin
// holds every block's candidate of column p, cout gets those of column p + 1, perm[p] the
// pivot row; *bad is set where a pivot vanishes or is not finite.  p = -1 only finds the
// first candidates.  A step is a chain of three trips to L2 (candidates, pivot row, rows);
// a row is loaded whole while the candidates are compared, and the one division is done by
// one warp (a division by every thread costs as much as the update).
template <int NV>
__global__ void __launch_bounds__(32 * GJ_W) k_gj_step(int n, int p, const double* in_, double* out,
                                                       const GjCand* cin_, GjCand* cout, int* perm, int* bad) {
  chained();
  const double* const in = fresh(in_);
  const GjCand* const cin = fresh(cin_);
  __shared__ double rp[32 * NV];  // the scaled pivot row
  __shared__ double inv_s;
  __shared__ int q_s;
  __shared__ GjCand cand[GJ_W];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, i = blockIdx.x * GJ_W + w;
  double v[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = i < n && 32 * k + lane < n ? in[(size_t)i * n + 32 * k + lane] : 0.0;
  if (p >= 0) {
    if (w == 0) {
      double c = 0.0;
      int row = n;
      bool nan = false;
      for (int b = lane; b < (int)gridDim.x; b += 32) {
        const GjCand x = cin[b];
        nan |= x.v != x.v;
        if (gj_before(x.v, x.row, c, row)) {
          c = x.v;
          row = x.row;
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double c2 = __shfl_xor_sync(0xffffffffu, c, o);
        const int r2 = __shfl_xor_sync(0xffffffffu, row, o);
        if (gj_before(c2, r2, c, row)) {
          c = c2;
          row = r2;
        }
      }
      nan = __any_sync(0xffffffffu, nan);
      const double inv = 1.0 / c;
      if (lane == 0) {
        inv_s = inv;
        q_s = row < n ? row : p;
        if (blockIdx.x == 0) {
          perm[p] = q_s;
          if (nan || c == 0.0 || !isfinite(c)) *bad = 1;
        }
      }
    }
    __syncthreads();
    const int q = q_s;
    const double inv = inv_s;
    for (int j = threadIdx.x; j < n; j += 32 * GJ_W) rp[j] = (j == p ? 1.0 : in[(size_t)q * n + j]) * inv;
    if (i == q && q != p) {  // the row that the interchange puts here
#pragma unroll
      for (int k = 0; k < NV; ++k) v[k] = 32 * k + lane < n ? in[(size_t)p * n + 32 * k + lane] : 0.0;
    }
    __syncthreads();
    const double f = i < n ? in[(size_t)(i == q ? p : i) * n + p] : 0.0;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const int j = 32 * k + lane;
      if (j < n) v[k] = i == p ? rp[j] : (j == p ? 0.0 : v[k]) - f * rp[j];
    }
    if (i < n) {
#pragma unroll
      for (int k = 0; k < NV; ++k)
        if (32 * k + lane < n) out[(size_t)i * n + 32 * k + lane] = v[k];
    }
  }
  if (lane == 0) cand[w] = GjCand{0.0, n, 0};
  __syncwarp();
  if (p + 1 < n && i < n && i >= p + 1) {
#pragma unroll
    for (int k = 0; k < NV; ++k)
      if (32 * k + lane == p + 1) cand[w] = GjCand{v[k], i, 0};
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    GjCand best = cand[0];
    for (int k = 1; k < GJ_W; ++k)
      if (cand[k].v != cand[k].v || gj_before(cand[k].v, cand[k].row, best.v, best.row)) best = cand[k];
    cout[blockIdx.x] = best;
  }
}

// Column of the eliminated matrix that each column of the inverse is: the row
// interchanges undone as column interchanges, in reverse order.
__global__ void k_gj_columns(int n, const int* perm_, int* map) {
  chained();
  const int* const perm = fresh(perm_);
  extern __shared__ int m[];
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    m[j] = j;
    m[n + j] = perm[j];
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int p = n - 1; p >= 0; --p) {
      const int q = m[n + p], t = m[p];
      m[p] = m[q];
      m[q] = t;
    }
  __syncthreads();
  for (int j = threadIdx.x; j < n; j += blockDim.x) map[j] = m[j];
}

// The inverse and its transpose in the cycle's precision.
template <typename R>
__global__ void k_gj_store(int n, const double* A_, const int* map_, R* inv) {
  chained();
  const double* const A = fresh(A_);
  const int* const map = fresh(map_);
  const int j = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y;
  if (j >= n) return;
  const R v = R(A[(size_t)i * n + map[j]]);
  inv[(size_t)i * n + j] = v;
  inv[(size_t)n * n + (size_t)j * n + i] = v;
}

// T = A^T (row-major n x n).  On the host this and the second half of the upload made a
// linearisation 0.1 ms longer at n = 320.
template <typename R>
__global__ void k_transposed(int n, const R* __restrict__ A, R* __restrict__ T) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y;
  if (j < n) T[(size_t)j * n + i] = A[(size_t)i * n + j];
}

// Smallest system inverted on the device.  The device pays 7 to 9 us a pivot (launch and
// three trips to L2; 2.2 us of it are the n^2 operations at n = 1000), one core 2 n^3
// operations out of its cache.  Linearisation of a one-level hierarchy, host / device:
// n = 320 1.2 / 2.2 ms, 400 2.0 / 2.8, 500 4.5 / 3.6, 560 5.6 / 4.6, 750 18 / 6.7,
// 1000 46 / 10.8 ms.
constexpr int GJ_DEVICE_MIN = 480;
static_assert(COARSE_DENSE_MAX <= 32 * 32, "a lane of k_gj_step holds at most 32 entries of a row");

// inv_dev <- the inverse of the host matrix A (overwritten) and its transpose.
template <typename R>
nc_status invert(nc_ctx* ctx, std::vector<double>& A, int n, R* inv_dev, const char* singular, cudaStream_t s) {
  nc_status st;
  if (n >= GJ_DEVICE_MIN) {
    const int blocks = (n + GJ_W - 1) / GJ_W;
    const size_t nn = (size_t)n * n, need = sizeof(double) * 2 * nn + sizeof(GjCand) * 2 * blocks +
                                            sizeof(int) * (2 * (size_t)n + 1);
    if (ctx->gj_bytes < need) {
      void* p = nullptr;
      if (cudaMalloc(&p, need) == cudaSuccess) {
        cudaFree(ctx->gj);
        ctx->gj = p;
        ctx->gj_bytes = need;
      } else {
        cudaGetLastError();  // no room: on the host below
      }
    }
    if (ctx->gj_bytes >= need) {
      double* M[2] = {(double*)ctx->gj, (double*)ctx->gj + nn};
      GjCand* C[2] = {(GjCand*)(M[1] + nn), (GjCand*)(M[1] + nn) + blocks};
      int *perm = (int*)(C[1] + blocks), *map = perm + n, *bad = map + n;
      cudaMemsetAsync(bad, 0, sizeof(int), s);
      if ((st = cuda_check(ctx, cudaMemcpyAsync(M[0], A.data(), sizeof(double) * nn, cudaMemcpyHostToDevice, s),
                           "coarse H2D")) != NC_OK)
        return st;
      const auto step = n <= 512 ? k_gj_step<16> : k_gj_step<32>;
      for (int p = -1; p < n; ++p) {
        const int a = p & 1, b = (p + 1) & 1;  // step -1 leaves its candidates in C[0]
        launch(step, blocks, 32 * GJ_W, 0, s, n, p, p < 0 ? M[0] : M[a], M[b], C[a], C[b], perm, bad);
      }
      launch(k_gj_columns, 1, 256, 2 * sizeof(int) * n, s, n, perm, map);
      launch(k_gj_store<R>, dim3((n + 255) / 256, n), 256, 0, s, n, M[n & 1], map, inv_dev);
      int h = 0;
      if ((st = cuda_check(ctx, cudaMemcpyAsync(&h, bad, sizeof(int), cudaMemcpyDeviceToHost, s),
                           "coarse inverse")) != NC_OK ||
          (st = cuda_check(ctx, cudaStreamSynchronize(s), "coarse sync")) != NC_OK)
        return st;
      return h ? set_err(ctx, NC_ERR_NAN, singular) : NC_OK;
    }
  }
  if (!gauss_jordan_inverse(A, n)) return set_err(ctx, NC_ERR_NAN, singular);
  const std::vector<R> Ar(A.begin(), A.end());
  if ((st = cuda_check(ctx, cudaMemcpyAsync(inv_dev, Ar.data(), sizeof(R) * Ar.size(),
                                            cudaMemcpyHostToDevice, s), "coarse H2D")) != NC_OK)
    return st;
  k_transposed<R><<<dim3((n + 255) / 256, n), 256, 0, s>>>(n, inv_dev, inv_dev + (size_t)n * n);
  return cuda_check(ctx, cudaStreamSynchronize(s), "coarse sync");
}

}  // namespace

int coarse_dense_dofs(const Level& L) { return (int)(5 * L.d.Nn); }

template <typename R>
nc_status coarse_setup(nc_ctx* ctx, Level& L, const R* x, const R* gam, const R* src,
                       R** inv_dev, cudaStream_t s) {
  const int n = coarse_dense_dofs(L);
  const long long E = L.d.E;
  nc_status st;
  if (ctx->cjel_elems < E) {
    cudaFree(ctx->cjel);
    ctx->cjel = nullptr;
    ctx->cjel_elems = 0;
    if ((st = cuda_check(ctx, cudaMalloc((void**)&ctx->cjel, sizeof(double) * 1600 * E),
                         "cudaMalloc coarse")) != NC_OK)
      return st;
    ctx->cjel_elems = E;
  }
  if (!*inv_dev) {
    if ((st = cuda_check(ctx, cudaMalloc((void**)inv_dev, sizeof(R) * 2 * (size_t)n * n),
                         "cudaMalloc coarse inverse")) != NC_OK)
      return st;
  }
  k_coarse_elem_jac<R><<<(unsigned)E, 64, 0, s>>>(L.d, L.c64, x, gam, src, ctx->cjel);
  std::vector<double> jel((size_t)1600 * E);
  std::vector<uint8_t> fl((size_t)L.d.Nn);
  if ((st = cuda_check(ctx, cudaMemcpyAsync(jel.data(), ctx->cjel, sizeof(double) * jel.size(),
                                            cudaMemcpyDeviceToHost, s), "coarse D2H")) != NC_OK ||
      (st = cuda_check(ctx, cudaMemcpyAsync(fl.data(), L.flag, fl.size(), cudaMemcpyDeviceToHost, s),
                       "coarse flags D2H")) != NC_OK ||
      (st = cuda_check(ctx, cudaStreamSynchronize(s), "coarse sync")) != NC_OK)
    return st;
  // dense assembly, unknown index f * Nn + node
  const LevelDev& d = L.d;
  const long long Nn = d.Nn;
  std::vector<double> A((size_t)n * n, 0.0);
  const long long sy = d.nx + 1, sz = (long long)(d.nx + 1) * (d.ny + 1);
  for (long long e = 0; e < E; ++e) {
    int i, j, kk;
    elem_ijk(d, e, i, j, kk);
    const long long n0 = i + sy * (j + (long long)(d.ny + 1) * kk);
    long long nodes[8];
    for (int a = 0; a < 8; ++a) nodes[a] = n0 + (a & 1) + ((a >> 1) & 1) * sy + ((a >> 2) & 1) * sz;
    for (int k = 0; k < 40; ++k) {
      const long long col = (k / 8) * Nn + nodes[k % 8];
      const double* cj = &jel[(size_t)(e * 40 + k) * 40];
      for (int r = 0; r < 40; ++r) {
        const long long row = (r / 8) * Nn + nodes[r % 8];
        A[(size_t)row * n + col] += cj[r];
      }
    }
  }
  for (long long node = 0; node < Nn; ++node)
    for (int f = 0; f < 5; ++f)
      if ((fl[node] >> f) & 1) {
        const long long r = f * Nn + node;
        for (int c = 0; c < n; ++c) A[(size_t)r * n + c] = 0.0;
        A[(size_t)r * n + r] = 1.0;
      }
  return invert(ctx, A, n, *inv_dev, "coarsest-level operator is singular", s);
}

template <typename R>
nc_status coarse_setup_stencil(nc_ctx* ctx, Level& L, const R* S, R** inv_dev, cudaStream_t s) {
  const int n = coarse_dense_dofs(L);
  const LevelDev& d = L.d;
  const long long Nn = d.Nn;
  nc_status st;
  if (!*inv_dev) {
    if ((st = cuda_check(ctx, cudaMalloc((void**)inv_dev, sizeof(R) * 2 * (size_t)n * n),
                         "cudaMalloc coarse inverse")) != NC_OK)
      return st;
  }
  std::vector<R> sh((size_t)STENCIL_VALUES * Nn);
  if ((st = cuda_check(ctx, cudaMemcpyAsync(sh.data(), S, sizeof(R) * sh.size(),
                                            cudaMemcpyDeviceToHost, s), "coarse stencil D2H")) != NC_OK ||
      (st = cuda_check(ctx, cudaStreamSynchronize(s), "coarse sync")) != NC_OK)
    return st;
  // dense assembly, unknown index f * Nn + node; Dirichlet rows are identity rows
  // of the stencil already
  std::vector<double> A((size_t)n * n, 0.0);
  for (long long node = 0; node < Nn; ++node) {
    int i, j, k;
    node_ijk(d, node, i, j, k);
    for (int o = 0; o < 27; ++o) {
      const int ii = i + o % 3 - 1, jj = j + (o / 3) % 3 - 1, kk = k + o / 9 - 1;
      if (ii < 0 || ii > d.nx || jj < 0 || jj > d.ny || kk < 0 || kk > d.nz) continue;
      const long long m = ii + (long long)(d.nx + 1) * (jj + (long long)(d.ny + 1) * kk);
      for (int f = 0; f < 5; ++f)
        for (int g = 0; g < 5; ++g)
          A[(size_t)(f * Nn + node) * n + (g * Nn + m)] =
              (double)sh[(size_t)((o * 5 + f) * 5 + g) * Nn + node];
    }
  }
  return invert(ctx, A, n, *inv_dev, "coarsest-level Galerkin operator is singular", s);
}

template <typename R>
void coarse_apply(const Level& L, bool tr, const R* inv, const R* b, R* z, cudaStream_t s) {
  const int n = coarse_dense_dofs(L);
  k_dense_gemv<R><<<(n + 7) / 8, 256, 0, s>>>(n, tr ? inv + (size_t)n * n : inv, b, z);
}

template nc_status coarse_setup<double>(nc_ctx*, Level&, const double*, const double*,
                                        const double*, double**, cudaStream_t);
template nc_status coarse_setup<float>(nc_ctx*, Level&, const float*, const float*, const float*,
                                       float**, cudaStream_t);
template void coarse_apply<double>(const Level&, bool, const double*, const double*, double*,
                                   cudaStream_t);
template nc_status coarse_setup_stencil<double>(nc_ctx*, Level&, const double*, double**,
                                                cudaStream_t);
template nc_status coarse_setup_stencil<float>(nc_ctx*, Level&, const float*, float**,
                                               cudaStream_t);
template void coarse_apply<float>(const Level&, bool, const float*, const float*, float*,
                                  cudaStream_t);

}  // namespace nc
