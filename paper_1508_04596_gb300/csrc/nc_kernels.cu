// Element operators, assembly by node-owner gather, and grid transfers.
//
// Assembly is colouring-free and deterministic: the element kernels write sums per
// node and element layer (the marching operators, nc_march.cuh) or 40 rows per element
// (diag(J)) to a scratch array, and one thread per node adds those of its node in a
// fixed order; the assembled Jacobian takes one contribution per entry and launch
// (nc_assemble.cuh).  Results are bitwise reproducible.
#include <type_traits>

#include "nc_assemble.cuh"
#include "nc_element_f2.cuh"
#include "nc_internal.cuh"
#include "nc_march.cuh"
#include "nc_reduce.cuh"
#include "nc_split.cuh"
#include "nc_transfer.cuh"

namespace nc {

namespace {

constexpr int ELEM_THREADS = 128;
constexpr int NODE_THREADS = 256;
constexpr unsigned PROLONG_BLOCKS = 8 * 152;  // blocks that fill the GPU: a thread per node from here

inline unsigned nblocks(long long n, int t) { return (unsigned)((n + t - 1) / t); }


__device__ __forceinline__ long long node_id(const LevelDev& d, int i, int j, int k) {
  return i + (long long)(d.nx + 1) * (j + (long long)(d.ny + 1) * k);
}

template <typename R>
__device__ __forceinline__ void load_elem(const LevelDev& d, const R* __restrict__ x, long long e,
                                          R xe[5][8], bool mask) {
  int i, j, k;
  elem_ijk(d, e, i, j, k);
  const long long n0 = node_id(d, i, j, k);
  const long long sy = d.nx + 1, sz = (long long)(d.nx + 1) * (d.ny + 1);
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const long long n = n0 + (a & 1) + ((a >> 1) & 1) * sy + ((a >> 2) & 1) * sz;
    const uint8_t fl = mask ? d.flag[n] : uint8_t(0);
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      R v = x[f * d.Nn + n];
      xe[f][a] = (fl >> f) & 1 ? R(0) : v;
    }
  }
}

// node of local index a (bit 0: +x, bit 1: +y, bit 2: +z) of element e
__device__ __forceinline__ long long elem_node(const LevelDev& d, long long e, int a) {
  int i, j, k;
  elem_ijk(d, e, i, j, k);
  return node_id(d, i + (a & 1), j + ((a >> 1) & 1), k + ((a >> 2) & 1));
}

// first row of element e in the blocked scratch; row r = 8 f + a is at + r YB
__device__ __forceinline__ long long yrow0(long long e) {
  static_assert(YB == 32, "yrow0 takes the block by a shift");
  return (e >> 5) * (40 * YB) + (e & (YB - 1));  // e >= 0
}

template <typename R>
__device__ __forceinline__ void store_elem(long long E, long long e, const R out[5][8], R* Y) {
  (void)E;
  R* y = Y + yrow0(e);
#pragma unroll
  for (int f = 0; f < 5; ++f)
#pragma unroll
    for (int a = 0; a < 8; ++a) y[(f * 8 + a) * YB] = out[f][a];
}

// Column col = 5 b + g of every element Jacobian: the element product with the
// unit direction on unknown g of local node b, or zero where that unknown is
// Dirichlet (Dirichlet columns are removed).  Re-interpolates the state: the way
// to assemble in FP32 where there is no memory for a linearisation store.
__global__ void __launch_bounds__(ELEM_THREADS) k_elem_column(
    LevelDev d, ElemConst<float> c, const float* __restrict__ x, const float* __restrict__ gam,
    const float* __restrict__ src, int col, float* Y) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= d.E) return;
  const int b = col / 5, g = col % 5;
  float out[5][8];
  if ((d.flag[elem_node(d, e, b)] >> g) & 1) {
#pragma unroll
    for (int f = 0; f < 5; ++f)
#pragma unroll
      for (int a = 0; a < 8; ++a) out[f][a] = 0.0f;
    store_elem(d.E, e, out, Y);
    return;
  }
  float ve[5][8], xe[5][8];
#pragma unroll
  for (int f = 0; f < 5; ++f)
#pragma unroll
    for (int a = 0; a < 8; ++a) ve[f][a] = (f == g && a == b) ? 1.0f : 0.0f;
  load_elem(d, x, e, xe, false);
  elem_jvp<float>(xe, ve, gam[e], src ? src[e] : 0.0f, c, out);
  store_elem(d.E, e, out, Y);
}

// S += column col = 5 b + g of the element Jacobians, summed per node: row (n, f)
// takes entry (f, a) of each element e around n (n is e's local node a), at the
// stencil offset of e's local node b from n.  The eight elements around n give
// eight distinct offsets, so one launch writes no entry twice; the launches run
// in column order, so the sums are deterministic.  Dirichlet rows are skipped
// (they become identity rows afterwards).
__global__ void __launch_bounds__(NODE_THREADS) k_assemble_column(LevelDev d, int col,
                                                                  const float* __restrict__ Y,
                                                                  float* __restrict__ S) {
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= d.Nn) return;
  int i, j, k;
  node_ijk(d, n, i, j, k);
  const int b = col / 5, g = col % 5;
  const uint8_t fl = d.flag[n];
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const int ie = i - (a & 1), je = j - ((a >> 1) & 1), ke = k - ((a >> 2) & 1);
    if (ie < 0 || je < 0 || ke < 0 || ie >= d.nx || je >= d.ny || ke >= d.nz) continue;
    const long long e = ie + (long long)d.nx * (je + (long long)d.ny * ke);
    const int o = ((b & 1) - (a & 1) + 1) + 3 * (((b >> 1) & 1) - ((a >> 1) & 1) + 1) +
                  9 * (((b >> 2) & 1) - ((a >> 2) & 1) + 1);
#pragma unroll
    for (int f = 0; f < 5; ++f)
      if (!((fl >> f) & 1)) S[((long long)(o * 5 + f) * 5 + g) * d.Nn + n] += Y[yrow0(e) + (f * 8 + a) * YB];
  }
}

template <typename R>
__global__ void __launch_bounds__(ELEM_THREADS) k_elem_diag(LevelDev d, ElemConst<R> c,
                                                            const R* __restrict__ x,
                                                            const R* __restrict__ gam,
                                                            const R* __restrict__ src, R* Y) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= d.E) return;
  R xe[5][8], out[5][8];
  load_elem(d, x, e, xe, false);
  elem_diag<R>(xe, gam[e], src ? src[e] : R(0), c, out);
  store_elem(d.E, e, out, Y);
}

enum GatherMode { G_RES = 0, G_LIN = 1, G_DIAG = 2 };

__device__ __forceinline__ int patch_face_count(const LevelDev& d, int i, int j, int k) {
  if (d.patch_mode != NC_PATCH_FLUX || k != 0) return 0;
  int cnt = 0;
#pragma unroll
  for (int di = -1; di <= 0; ++di)
#pragma unroll
    for (int dj = -1; dj <= 0; ++dj) {
      const int ie = i + di, je = j + dj;
      cnt += (ie >= d.pi0 && ie <= d.pi1 - 1 && je >= d.pj0 && je <= d.pj1 - 1) ? 1 : 0;
    }
  return cnt;
}

// Row values of node n from the sums acc of its elements: Dirichlet rows, patch flux.
template <typename R, int MODE>
__device__ __forceinline__ void node_rows(const LevelDev& d, long long n, int i, int j, int k, R acc[5],
                                          const R* __restrict__ xv, R* __restrict__ out) {
  const uint8_t fl = d.flag[n];
  if (MODE == G_RES) {
    const int pc = patch_face_count(d, i, j, k);
    if (pc) acc[4] -= R(d.q * d.h * d.h * 0.25 * pc);
  }
#pragma unroll
  for (int f = 0; f < 5; ++f) {
    R v = acc[f];
    if ((fl >> f) & 1) {
      if (MODE == G_RES) {
        const R xd = (f == 4) ? R(d.tval[fl >> 5]) : R(0);
        v = xv[f * d.Nn + n] - xd;
      } else if (MODE == G_LIN) {
        v = xv[f * d.Nn + n];
      } else {
        v = R(1);
      }
    }
    out[f * d.Nn + n] = v;
  }
}

// Gather of the 40 element rows (diag(J)).
template <typename R, int MODE>
__global__ void __launch_bounds__(NODE_THREADS) k_gather(LevelDev d, const R* __restrict__ Y,
                                                         const R* __restrict__ xv, R* out) {
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= d.Nn) return;
  int i, j, k;
  node_ijk(d, n, i, j, k);
  R acc[5] = {R(0), R(0), R(0), R(0), R(0)};
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const int ie = i - (a & 1), je = j - ((a >> 1) & 1), ke = k - ((a >> 2) & 1);
    if (ie < 0 || je < 0 || ke < 0 || ie >= d.nx || je >= d.ny || ke >= d.nz) continue;
    const long long e = ie + (long long)d.nx * (je + (long long)d.ny * ke);
#pragma unroll
    for (int f = 0; f < 5; ++f) acc[f] += Y[yrow0(e) + (f * 8 + a) * YB];
  }
  node_rows<R, MODE>(d, n, i, j, k, acc, xv, out);
}

// Gather of the marching kernels' sums.
template <typename R, int MODE>
__global__ void __launch_bounds__(NODE_THREADS) k_gather_march(LevelDev d, MarchPlan mp,
                                                               const R* __restrict__ Y_,
                                                               const R* __restrict__ xv_,
                                                               const R* __restrict__ b_,
                                                               R* __restrict__ out) {
  chained();
  const R* const Y = fresh(Y_);
  const R* const xv = fresh(xv_);
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= d.Nn) return;
  int i, j, k;
  node_ijk(d, n, i, j, k);
  R acc[5] = {R(0), R(0), R(0), R(0), R(0)};
  march::node_sums(d, mp, i, j, k, Y, acc);
  if (MODE == G_LIN && b_) {  // b - A v
    const R* const b = fresh(b_);
    const uint8_t fl = d.flag[n];
#pragma unroll
    for (int f = 0; f < 5; ++f)
      out[f * d.Nn + n] = b[f * d.Nn + n] - ((fl >> f) & 1 ? xv[f * d.Nn + n] : acc[f]);
    return;
  }
  node_rows<R, MODE>(d, n, i, j, k, acc, xv, out);
}

// The same for a product w = A v with the dots <V_q, w>, q < k <= KB, that the smoother
// takes of it next: the result is not read back, and no multi-dot is launched (a third
// of the reduction launches; on a small level a launch costs more than its work).
// Two accumulators per column; partials fold in the last block.
// TH threads a block: 1024 where one block holds every node (nothing to fold then).
template <typename R, int KB, int TH>
__global__ void __launch_bounds__(TH) k_gather_dots(LevelDev d, MarchPlan mp,
                                                              const R* __restrict__ Y_,
                                                              const R* __restrict__ xv_,
                                                              R* __restrict__ out, int k,
                                                              const R* __restrict__ V_, long long ld,
                                                              double* partial, double* dots,
                                                              const double* sig2, double* cf,
                                                              unsigned* ticket) {
  chained();
  const R* const Y = fresh(Y_);
  const R* const xv = fresh(xv_);
  const R* const V = fresh(V_);
  R a0[KB], a1[KB];
#pragma unroll
  for (int q = 0; q < KB; ++q) a0[q] = a1[q] = R(0);
  for (long long n = blockIdx.x * (long long)TH + threadIdx.x; n < d.Nn;
       n += (long long)gridDim.x * TH) {
    int i, j, kk;
    node_ijk(d, n, i, j, kk);
    R acc[5] = {R(0), R(0), R(0), R(0), R(0)};
    march::node_sums(d, mp, i, j, kk, Y, acc);
    const uint8_t fl = d.flag[n];
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      const R w = (fl >> f) & 1 ? xv[f * d.Nn + n] : acc[f];
      out[f * d.Nn + n] = w;
      acc[f] = w;
    }
#pragma unroll
    for (int q = 0; q < KB; ++q)
      if (q < k) {
        const R* p = V + q * ld + n;
        R u[5];
#pragma unroll
        for (int f = 0; f < 5; ++f) u[f] = p[f * d.Nn];
        a0[q] = fma(u[0], acc[0], fma(u[2], acc[2], fma(u[4], acc[4], a0[q])));
        a1[q] = fma(u[1], acc[1], fma(u[3], acc[3], a1[q]));
      }
  }
  R v[KB];
#pragma unroll
  for (int q = 0; q < KB; ++q) v[q] = q < k ? a0[q] + a1[q] : R(0);
  block_values<TH>(v, k, partial);
  if (last_block(ticket))
    fold_values(k, gridDim.x, partial, [&](int q, double t) {
      dots[q] = t;
      cf[q] = coef_over(t, sig2[q]);
    });
}

template <typename R, bool ZERO>
__global__ void k_impose(LevelDev d, R* x) {
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= d.Nn) return;
  const uint8_t fl = d.flag[n];
  if (!(fl & 31)) return;
#pragma unroll
  for (int f = 0; f < 5; ++f)
    if ((fl >> f) & 1) x[f * d.Nn + n] = (f == 4 && !ZERO) ? R(d.tval[fl >> 5]) : R(0);
}

__global__ void k_objective_grad(LevelDev d, double* g, double inv_area) {
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= (long long)(d.nx + 1) * (d.ny + 1)) return;  // bottom plane only
  const int i = (int)(n % (d.nx + 1));
  const int j = (int)(n / (d.nx + 1));
  int cnt = 0;
  for (int di = -1; di <= 0; ++di)
    for (int dj = -1; dj <= 0; ++dj) {
      const int ie = i + di, je = j + dj;
      cnt += (ie >= d.pi0 && ie <= d.pi1 - 1 && je >= d.pj0 && je <= d.pj1 - 1) ? 1 : 0;
    }
  g[4 * d.Nn + n] = cnt * d.h * d.h * 0.25 * inv_area;
}

// Gradient of the thermal compliance f = int s T dV: T rows get
// sum over the node's elements of s_e h^3 / 8 (int_e N_a dV = h^3/8), in a fixed
// element order.
__global__ void k_source_grad(LevelDev d, const double* __restrict__ src, double* g) {
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= d.Nn) return;
  int i, j, k;
  node_ijk(d, n, i, j, k);
  double acc = 0.0;
  for (int a = 0; a < 8; ++a) {
    const int ie = i - (a & 1), je = j - ((a >> 1) & 1), ke = k - ((a >> 2) & 1);
    if (ie < 0 || je < 0 || ke < 0 || ie >= d.nx || je >= d.ny || ke >= d.nz) continue;
    acc += src[ie + (long long)d.nx * (je + (long long)d.ny * ke)];
  }
  g[4 * d.Nn + n] = acc * d.h * d.h * d.h * 0.125;
}

// A thread per node and field (blockIdx.y): with a thread per node the coarse levels
// are too few threads to hide the latency of 27 x 5 loads (64^3 -> 32^3: 21 us, 9 now),
// and on fine ones its registers leave too few warps (192x192x384 429 us, 246).
template <typename R>
__global__ void k_restrict(LevelDev f, const R* __restrict__ rf, LevelDev c, R* __restrict__ rc) {
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= c.Nn) return;
  const int q = blockIdx.y;
  int I, J, K;
  node_ijk(c, n, I, J, K);
  rc[q * c.Nn + n] = restrict_value(f, rf + q * f.Nn, q, c.flag[n], I, J, K);
}

// A thread per node with Q = 5, per node and field (blockIdx.y) with Q = 1: where the
// nodes fill the GPU, five threads only repeat the index arithmetic and the branches
// (192x192x384 482 us, 266 with a thread per node; 96x96x192 63 and 36).
template <typename R, int Q>
__global__ void k_prolong_add(LevelDev c, const R* __restrict__ zc, LevelDev f, R* __restrict__ zf) {
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= f.Nn) return;
  int i, j, k;
  node_ijk(f, n, i, j, k);
  const uint8_t fl = f.flag[n];
  R v[Q], z[Q];
#pragma unroll
  for (int u = 0; u < Q; ++u) {
    const int q = Q * blockIdx.y + u;
    z[u] = zf[q * f.Nn + n];
    v[u] = prolong_value(c, zc + q * c.Nn, i, j, k);
  }
#pragma unroll
  for (int u = 0; u < Q; ++u) {
    const int q = Q * blockIdx.y + u;
    if (!((fl >> q) & 1)) zf[q * f.Nn + n] = z[u] + v[u];
  }
}

template <typename R>
__global__ void k_inject(LevelDev f, const R* __restrict__ xf, LevelDev c, R* xc) {
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= c.Nn) return;
  int I, J, K;
  node_ijk(c, n, I, J, K);
  const long long m = node_id(f, 2 * I, 2 * J, 2 * K);
#pragma unroll
  for (int q = 0; q < 5; ++q) xc[q * c.Nn + n] = xf[q * f.Nn + m];
}

template <typename R>
__global__ void k_coarsen_elem(LevelDev f, const R* __restrict__ gf, LevelDev c, R* gc) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= c.E) return;
  int I, J, K;
  elem_ijk(c, e, I, J, K);
  R acc = R(0);
  for (int a = 0; a < 8; ++a) {
    const int i = 2 * I + (a & 1), j = 2 * J + ((a >> 1) & 1), k = 2 * K + ((a >> 2) & 1);
    acc += gf[i + (long long)f.nx * (j + (long long)f.ny * k)];
  }
  gc[e] = acc * R(0.125);
}

}  // namespace

// Chunks of 31 faces share their end faces; 32 where a layer's row of faces divides 32
// and no element straddles two chunks.  The run length is the one that takes the
// fewest steps on the busiest scheduler.  FP32 kernels are bound by latency at 8 warps
// on each of 152 SMs, which finish a run in about the time one takes; a run of rc rows
// costs its steps and 0.6 of one for the first row's loads and the extra row of sums.
// FP64 steps pass the 608 schedulers' FP64 units one after the other, so there the
// runs per scheduler count.  (96^3: FP32 J v 119, 92, 86, 84 us with runs of 1, 4, 8, 24
// rows; 64^3, FP64 J v from the store: 680, 703, 673, 694, 683, 811 us with 1 to 6.)  Runs
// of several rows are taken only where their sums fit the element-row scratch; single
// rows, cut into chunks all together, always do: 640 values per 31 faces (2 rows of 10
// sums per lane) against 40 per element, or per 32 faces with one element across.
MarchPlan march_plan(const LevelDev& d, bool fp64) {
  const long long slots = fp64 ? 608 : 8 * 152;
  const double extra = fp64 ? 0.05 : 0.6;
  MarchPlan p;
  p.stride = 32 % (d.nx + 1) == 0 ? 32 : 31;
  const long long faces = (long long)(d.nx + 1) * d.nz;
  p.flat = 1;
  p.rc = 1;
  p.runs = d.ny;
  p.nchunk = (faces * d.ny + p.stride - 1) / p.stride;
  auto steps = [&](const MarchPlan& m) {  // a lone run per FP64 unit hides no latency
    const long long turns = (m.warps() + slots - 1) / slots;
    return (m.rc + extra) * (fp64 && turns == 1 ? 1.12 : (double)turns);
  };
  double cost = steps(p);
  MarchPlan q = p;
  q.flat = 0;
  q.nchunk = (faces + p.stride - 1) / p.stride;
  for (q.rc = 2; q.rc <= 24 && q.rc <= d.ny; ++q.rc) {
    q.runs = (d.ny + q.rc - 1) / q.rc;
    const double t = steps(q);
    if (t < cost && q.scratch() <= scratch_len(d.E)) {
      cost = t;
      p = q;
    }
  }
  // Four warps per chunk while that keeps the schedulers short of work (FP64: at most two
  // chunks' quarters each): residual FP64 at 12^3 27 us against 51, at 20^3 39 against
  // 51, at 24^3 68 against 51; FP32 J v 10.3 against 12.4 at 16^3, even at 32^3.
  p.split = p.flat && p.nchunk <= (fp64 ? 304 : 750);
  return p;
}

// A warp for every chunk of faces and run of rows, four to a block: one on each
// scheduler (blocks of one warp leave schedulers idle, FP64 23 % slower at 64^3).
template <typename R, int K>
static void run_march(const LevelDev& d, const ElemConst<R>& c, const R* x, const R* gam, const R* src,
                      const R* cache, const R* v, R* out, cudaStream_t s) {
  const MarchPlan mp = march_plan(d, sizeof(R) == 8);
  if constexpr (march::Traits<K>::TEST) {
    if (mp.split) {
      launch(march::k_split<R, K>, (unsigned)mp.nchunk, 128, 0, s, d, c, mp, x, gam, src, cache, v, out);
      return;
    }
  }
  launch(march::k_march<R, K>, nblocks(mp.warps(), march::WARPS), 32 * march::WARPS, 0, s, 
      d, c, mp, x, gam, src, cache, v, out);
}

template <typename R, int MODE>
static void run_gather(const LevelDev& d, const R* Y, const R* xv, R* out, cudaStream_t s,
                       const Dots<R>* dots = nullptr) {
  const MarchPlan mp = march_plan(d, sizeof(R) == 8);
  const unsigned nb = nblocks(d.Nn, NODE_THREADS);
  if (dots && dots->k > 0 && dots->k <= 8) {
    const unsigned rb = nb < RED_BLOCKS_MAX ? nb : RED_BLOCKS_MAX;
    auto go = [&](auto kernel, unsigned blocks, unsigned threads) {
      launch(kernel, blocks, threads, 0, s, d, mp, Y, xv, out, dots->k, dots->V, dots->ld, dots->partial,
             dots->out, dots->sig2, dots->cf, red_ticket(dots->partial));
    };
    if constexpr (sizeof(R) == 4) {
      if (nb > 1 && d.Nn <= 1024) {
        go(dots->k <= 4 ? k_gather_dots<R, 4, 1024> : k_gather_dots<R, 8, 1024>, 1, 1024);
        return;
      }
    }
    go(dots->k <= 4 ? k_gather_dots<R, 4, NODE_THREADS> : k_gather_dots<R, 8, NODE_THREADS>, rb, NODE_THREADS);
    return;
  }
  launch(k_gather_march<R, MODE>, nb, NODE_THREADS, 0, s, d, mp, Y, xv, dots ? dots->b : nullptr, out);
  if (dots && dots->k)
    vmdot_cf(5 * d.Nn, dots->k, dots->V, dots->ld, (const R*)out, dots->out, dots->sig2, dots->cf,
             dots->partial, s);
}

template <typename R>
void op_residual(const LevelDev& d, const ElemConst<R>& c, const R* x, const R* gam, const R* src,
                 R* r, R* Y, cudaStream_t s) {
  run_march<R, march::RES>(d, c, x, gam, src, nullptr, nullptr, Y, s);
  run_gather<R, G_RES>(d, Y, x, r, s);
}

template <typename R>
void op_jvp(const LevelDev& d, const ElemConst<R>& c, const R* x, const R* gam, const R* src,
            const R* v, R* out, R* Y, cudaStream_t s, const Dots<R>* dots) {
  run_march<R, march::JVP>(d, c, x, gam, src, nullptr, v, Y, s);
  run_gather<R, G_LIN>(d, Y, v, out, s, dots);
}

template <typename R>
void op_jtvp(const LevelDev& d, const ElemConst<R>& c, const R* x, const R* gam, const R* src,
             const R* w, R* out, R* Y, cudaStream_t s, const Dots<R>* dots) {
  run_march<R, march::JTVP>(d, c, x, gam, src, nullptr, w, Y, s);
  run_gather<R, G_LIN>(d, Y, w, out, s, dots);
}

template <typename R>
void op_linearize(const LevelDev& d, const ElemConst<R>& c, const R* x, const R* gam, const R* src,
                  R* cache, cudaStream_t s) {
  run_march<R, march::LINEARIZE>(d, c, x, gam, src, nullptr, nullptr, cache, s);
}

void op_jvp_cached(const LevelDev& d, const ElemConst<double>& c, const double* x, const double* gam,
                   const double* src, const double* cache, const double* v, double* out, double* Y,
                   cudaStream_t s, const Dots<double>* dots) {
  run_march<double, march::JVP_LIN>(d, c, x, gam, src, cache, v, Y, s);
  run_gather<double, G_LIN>(d, Y, v, out, s, dots);
}

void op_jtvp_cached(const LevelDev& d, const ElemConst<double>& c, const double* x, const double* gam,
                    const double* src, const double* cache, const double* w, double* out, double* Y,
                    cudaStream_t s, const Dots<double>* dots) {
  run_march<double, march::JTVP_LIN>(d, c, x, gam, src, cache, w, Y, s);
  run_gather<double, G_LIN>(d, Y, w, out, s, dots);
}

template <typename R>
void op_diag(const LevelDev& d, const ElemConst<R>& c, const R* x, const R* gam, const R* src,
             R* out, R* Y, cudaStream_t s) {
  k_elem_diag<R><<<nblocks(d.E, ELEM_THREADS), ELEM_THREADS, 0, s>>>(d, c, x, gam, src, Y);
  k_gather<R, G_DIAG><<<nblocks(d.Nn, NODE_THREADS), NODE_THREADS, 0, s>>>(d, Y, x, out);
}

template <typename R>
void op_assemble(const LevelDev& d, const ElemConst<R>& c, const R* x, const R* gam, const R* src,
                 const R* cache, R* S, R* Y, cudaStream_t s) {
  cudaMemsetAsync(S, 0, sizeof(R) * (size_t)STENCIL_VALUES * (size_t)d.Nn, s);
  if constexpr (sizeof(R) == 4) {
    if (!cache) {
      for (int col = 0; col < 40; ++col) {
        k_elem_column<<<nblocks(d.E, ELEM_THREADS), ELEM_THREADS, 0, s>>>(d, c, x, gam, src, col, Y);
        k_assemble_column<<<nblocks(d.Nn, NODE_THREADS), NODE_THREADS, 0, s>>>(d, col, Y, S);
      }
      stencil_dirichlet<R>(d, S, s);
      return;
    }
  }
  for (int a = 0; a < 8; ++a)
    rows::k_assemble_rows<R><<<nblocks(d.E, 128), 128, 0, s>>>(d, c, rows::row_const(c, a), x, cache, a, S);
  stencil_dirichlet<R>(d, S, s);
}

void op_sens(const LevelDev& d, const ElemConst<double>& c, const double* x, const double* gam,
             const double* src, const double* lam, double* out, cudaStream_t s) {
  run_march<double, march::SENS>(d, c, x, gam, src, nullptr, lam, out, s);
}

template <typename R>
void op_impose(const LevelDev& d, R* x, cudaStream_t s) {
  k_impose<R, false><<<nblocks(d.Nn, NODE_THREADS), NODE_THREADS, 0, s>>>(d, x);
}

template <typename R>
void op_mask(const LevelDev& d, R* x, cudaStream_t s) {
  k_impose<R, true><<<nblocks(d.Nn, NODE_THREADS), NODE_THREADS, 0, s>>>(d, x);
}

double patch_area(const LevelDev& d) {
  if (d.pi1 <= d.pi0 || d.pj1 <= d.pj0) return 0.0;
  return (double)(d.pi1 - d.pi0) * (double)(d.pj1 - d.pj0) * d.h * d.h;
}

void op_source_grad(const LevelDev& d, const double* src, double* g, cudaStream_t s) {
  cudaMemsetAsync(g, 0, sizeof(double) * 5 * d.Nn, s);
  k_source_grad<<<nblocks(d.Nn, NODE_THREADS), NODE_THREADS, 0, s>>>(d, src, g);
}

void op_objective_grad(const LevelDev& d, double* g, cudaStream_t s) {
  cudaMemsetAsync(g, 0, sizeof(double) * 5 * d.Nn, s);
  const double A = patch_area(d);
  if (A <= 0.0) return;
  const long long nb = (long long)(d.nx + 1) * (d.ny + 1);
  k_objective_grad<<<nblocks(nb, NODE_THREADS), NODE_THREADS, 0, s>>>(d, g, 1.0 / A);
}

template <typename R>
void op_restrict(const LevelDev& fine, const R* rf, const LevelDev& coarse, R* rc, cudaStream_t s) {
  k_restrict<R><<<dim3(nblocks(coarse.Nn, NODE_THREADS), NF), NODE_THREADS, 0, s>>>(fine, rf, coarse, rc);
}
template <typename R>
void op_prolong_add(const LevelDev& coarse, const R* zc, const LevelDev& fine, R* zf,
                    cudaStream_t s) {
  const unsigned nb = nblocks(fine.Nn, NODE_THREADS);
  if (nb >= PROLONG_BLOCKS)
    k_prolong_add<R, NF><<<nb, NODE_THREADS, 0, s>>>(coarse, zc, fine, zf);
  else
    k_prolong_add<R, 1><<<dim3(nb, NF), NODE_THREADS, 0, s>>>(coarse, zc, fine, zf);
}
template <typename R>
void op_inject(const LevelDev& fine, const R* xf, const LevelDev& coarse, R* xc, cudaStream_t s) {
  k_inject<R><<<nblocks(coarse.Nn, NODE_THREADS), NODE_THREADS, 0, s>>>(fine, xf, coarse, xc);
}
template <typename R>
void op_coarsen_elem(const LevelDev& fine, const R* gf, const LevelDev& coarse, R* gc,
                     cudaStream_t s) {
  k_coarsen_elem<R><<<nblocks(coarse.E, NODE_THREADS), NODE_THREADS, 0, s>>>(fine, gf, coarse, gc);
}

#define NC_INST(R)                                                                              \
  template void op_residual<R>(const LevelDev&, const ElemConst<R>&, const R*, const R*,        \
                               const R*, R*, R*, cudaStream_t);                                 \
  template void op_jvp<R>(const LevelDev&, const ElemConst<R>&, const R*, const R*, const R*,   \
                          const R*, R*, R*, cudaStream_t, const Dots<R>*);                      \
  template void op_jtvp<R>(const LevelDev&, const ElemConst<R>&, const R*, const R*, const R*,  \
                           const R*, R*, R*, cudaStream_t, const Dots<R>*);                     \
  template void op_diag<R>(const LevelDev&, const ElemConst<R>&, const R*, const R*, const R*,  \
                           R*, R*, cudaStream_t);                                               \
  template void op_linearize<R>(const LevelDev&, const ElemConst<R>&, const R*, const R*,       \
                                const R*, R*, cudaStream_t);                                    \
  template void op_assemble<R>(const LevelDev&, const ElemConst<R>&, const R*, const R*,        \
                               const R*, const R*, R*, R*, cudaStream_t);                       \
  template void op_impose<R>(const LevelDev&, R*, cudaStream_t);                                \
  template void op_mask<R>(const LevelDev&, R*, cudaStream_t);                                  \
  template void op_restrict<R>(const LevelDev&, const R*, const LevelDev&, R*, cudaStream_t);   \
  template void op_prolong_add<R>(const LevelDev&, const R*, const LevelDev&, R*, cudaStream_t);\
  template void op_inject<R>(const LevelDev&, const R*, const LevelDev&, R*, cudaStream_t);     \
  template void op_coarsen_elem<R>(const LevelDev&, const R*, const LevelDev&, R*, cudaStream_t);
NC_INST(double)
NC_INST(float)
#undef NC_INST

}  // namespace nc
