// PDE (Helmholtz) density filter (Sec. 3.2; filter radius 2.5 h in Sec. 6.3-6.4).
//
//   -r^2 lap(rho~) + rho~ = rho,  Neumann boundary,  r = R / (2 sqrt 3),
//
// with trilinear nodal rho~, element-constant rho, and the filtered element
// value the mean of its eight nodes: gamma~ = P rho, P = h^-3 T^T (r^2 K + M)^-1 T,
// T_{n,e} = int_e N_n = h^3/8.  P is symmetric, so the same call applies the
// chain rule dPhi/drho = P dPhi/dgamma~.
//
// On a uniform grid r^2 K + M is a sum of products of the 1-D stiffness and mass
// matrices.  Both have a boundary row that is half the interior row with the
// missing neighbour mirrored, so the operator is one symmetric 27-point stencil
// with four weights (by the number of coordinates that differ) on mirrored
// neighbours, halved once per boundary coordinate; its diagonal is a constant
// halved the same way.  The SPD system is solved by Jacobi-preconditioned
// conjugate gradients in FP64.
//
// An iteration is two kernels, and none waits for the host: alpha, beta and
// the stopping test are taken by the block that ends a reduction, and the host
// enqueues batches of iterations, fewer where it sees the end meanwhile (those after
// convergence return at once).
//  * k_cg_apply forms p = r / d + beta p on the fly while it loads its tile, then
//    q = A p and <p, q>: per plane, the four edge and four corner neighbours are
//    summed once and meet their weights afterwards, 15 FP64 operations per node and 2
//    per slot of the tile for p (23 per node with the halo), where a sum over the
//    eight elements takes 64;
//  * k_cg_update takes the steps of x and r with <r, r> and <r, r/d>, 5 per node.
// FP64 operations bound both (two FP64 lanes per SM): k_cg_apply keeps the pipe 78 % busy
// on the SMs that have a tile, k_cg_update, which waits for L2 as well, 70 %.  80x80x160
// (1.06M nodes, 19 iterations): 1.68 ms, k_cg_apply 58 us and k_cg_update 21 us an iteration; 5.75 ms
// with one kernel per vector operation, a 64-term product (146 us) and three host
// reads per iteration.
#include <algorithm>
#include <cmath>

#include "nc_internal.cuh"
#include "nc_reduce.cuh"

namespace nc {
nc_status set_err(nc_ctx* ctx, nc_status st, const std::string& msg);
nc_status cuda_check(nc_ctx* ctx, cudaError_t e, const char* what);
}  // namespace nc

using namespace nc;

namespace {

constexpr int FT = 256;

inline unsigned fblocks(long long n) { return (unsigned)((n + FT - 1) / FT); }

// Weights of the mirrored 27-point stencil by the number of coordinates in which the
// neighbour differs, and the reciprocal of the diagonal w[0] (interior values).
struct HelmCoef {
  double w[4], inv_d;
};

HelmCoef helm_coef(double h, double R) {
  const double r2 = R * R / 12.0;
  const double K[4] = {h / 3.0, 0.0, -h / 12.0, -h / 12.0};  // element stiffness entries
  const double M[4] = {8.0, 4.0, 2.0, 1.0};                  // element mass entries, x h^3/216
  const double elems[4] = {8.0, 4.0, 2.0, 1.0};              // elements that share both nodes
  HelmCoef c;
  for (int q = 0; q < 4; ++q) c.w[q] = elems[q] * (r2 * K[q] + M[q] * h * h * h / 216.0);
  c.inv_d = 1.0 / c.w[0];
  return c;
}

// State of one solve, on the device.
struct CgState {
  double bb, tol2, rr, rz, alpha, beta;
  int it, done;  // done: 0 running, 1 converged, 2 iteration limit, 3 non-finite input
  unsigned ticket, pad;
};
constexpr int CG_MAX_IT = 1000;

__device__ __forceinline__ int on_face(int i, int n) { return i == 0 || i == n; }
// 2^b, from the exponent bits (an integer conversion would take the FP64 pipe)
__device__ __forceinline__ double pow2(int b) { return __hiloint2double((1023 + b) << 20, 0); }

// b_n = sum over the node's elements of rho_e h^3 / 8; r = b, x = 0, <b, b>, <b, b/d>;
// whether there is nothing to solve goes to page-locked memory too.
__global__ void __launch_bounds__(FT) k_cg_rhs(LevelDev d, HelmCoef c, const double* __restrict__ rho,
                                               double* __restrict__ r, double* __restrict__ x,
                                               double* partial, CgState* s, int* host_done) {
  const double w = d.h * d.h * d.h * 0.125;
  double bb = 0.0, bz = 0.0;
  for (long long n = blockIdx.x * (long long)FT + threadIdx.x; n < d.Nn; n += (long long)gridDim.x * FT) {
    int i, j, k;
    node_ijk(d, n, i, j, k);
    double acc = 0.0;
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const int ie = i - (a & 1), je = j - ((a >> 1) & 1), ke = k - ((a >> 2) & 1);
      if (ie < 0 || je < 0 || ke < 0 || ie >= d.nx || je >= d.ny || ke >= d.nz) continue;
      acc += rho[ie + (long long)d.nx * (je + (long long)d.ny * ke)];
    }
    acc *= w;
    r[n] = acc;
    x[n] = 0.0;
    bb += acc * acc;
    bz += acc * acc * pow2(on_face(i, d.nx) + on_face(j, d.ny) + on_face(k, d.nz));
  }
  bb = block_fold<false, FT>(bb);
  if (threadIdx.x == 0) partial[blockIdx.x] = bb;
  bz = block_fold<false, FT>(bz);
  if (threadIdx.x == 0) partial[gridDim.x + blockIdx.x] = bz;
  if (!last_block(&s->ticket)) return;
  bb = fold_partials<false, FT>(gridDim.x, partial);
  bz = fold_partials<false, FT>(gridDim.x, partial + gridDim.x);
  if (threadIdx.x == 0) {
    s->bb = s->rr = bb;
    s->tol2 = 1e-26 * bb;  // ||r|| <= 1e-13 ||b||
    s->rz = bz * c.inv_d;
    s->beta = 0.0;
    s->it = 0;
    *host_done = s->done = !isfinite(bb) ? 3 : (bb > 0.0 ? 0 : 1);
  }
}

// Index of grid line position g, mirrored at both ends (and kept inside for the
// positions of a ragged tile that no owned node reads).
__device__ __forceinline__ int mirror(int g, int n) {
  g = g < 0 ? -g : (g > n ? 2 * n - g : g);
  return g < 0 ? 0 : (g > n ? n : g);
}

// p = r/d + beta p_old, q = A p, alpha = <r, r/d> / <p, q>.
// A block marches a tw x th node tile over zc planes; a plane of p with its halo is
// formed in shared memory (two buffers, one barrier per plane), the loads of the
// next plane in flight meanwhile.  P and Q are a plane's contributions to its own and
// to the adjacent planes' products.
constexpr int HSLOTS = 2 * FT;  // nodes of a tile with its halo at most
struct HelmTile {
  int tw, th, tiles_x, tiles_y, zc;
  long long items;  // tiles times marches
};
__global__ void __launch_bounds__(FT) k_cg_apply(LevelDev d, HelmCoef c, HelmTile t,
                                                 const double* __restrict__ r,
                                                 const double* __restrict__ p_old,
                                                 double* __restrict__ p_new, double* __restrict__ q,
                                                 double* partial, CgState* s) {
  if (s->done) return;
  const double beta = s->beta;
  const bool first = s->it == 0;  // p_old is not set yet
  __shared__ double sm[2][HSLOTS];
  const int tx = threadIdx.x % t.tw, ty = threadIdx.x / t.tw;
  const int hw = t.tw + 2, slots = hw * (t.th + 2);
  const long long sy = d.nx + 1, sz = (long long)(d.nx + 1) * (d.ny + 1);
  double pq = 0.0;
  for (long long item = blockIdx.x; item < t.items; item += gridDim.x) {
    const int bx = (int)(item % t.tiles_x), by = (int)(item / t.tiles_x % t.tiles_y);
    const int k0 = (int)(item / t.tiles_x / t.tiles_y) * t.zc, k1 = min(k0 + t.zc, d.nz + 1);
    long long at[2];  // node of the slot in plane 0
    double wxy[2], wxy2[2];  // 1/d on an inner and on a boundary plane
    bool own[2];      // the slot is a node of this tile
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int q = threadIdx.x + u * FT, sx = q % hw, s2 = q / hw;
      const int gi = bx * t.tw + sx - 1, gj = by * t.th + s2 - 1;
      const int mi = mirror(gi, d.nx), mj = mirror(gj, d.ny);
      at[u] = mi + sy * mj;
      wxy[u] = c.inv_d * pow2(on_face(mi, d.nx) + on_face(mj, d.ny));
      wxy2[u] = 2.0 * wxy[u];
      own[u] = sx >= 1 && sx <= t.tw && s2 >= 1 && s2 <= t.th && gi <= d.nx && gj <= d.ny;
    }
    const bool use[2] = {(int)threadIdx.x < slots, (int)threadIdx.x + FT < slots};
    const int i = bx * t.tw + tx, j = by * t.th + ty;
    const bool in = ty < t.th && i <= d.nx && j <= d.ny;
    const int faces_xy = on_face(i, d.nx) + on_face(j, d.ny);
    double rv[2] = {0.0, 0.0}, pv[2] = {0.0, 0.0};
    auto load = [&](int kk) {
      const long long off = sz * mirror(kk, d.nz);
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (use[u]) {
          rv[u] = r[at[u] + off];
          pv[u] = first ? 0.0 : p_old[at[u] + off];
        }
    };
    double P = 0.0, Q1 = 0.0, Q2 = 0.0, cp = 0.0;  // P, Q of plane kk - 1, Q of kk - 2, p of kk - 1
    load(k0 - 1);
    for (int kk = k0 - 1; kk <= k1; ++kk) {
      double* b = sm[kk & 1];
      const int gk = mirror(kk, d.nz);
      const bool face = on_face(gk, d.nz);
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (use[u]) {
          const double v = rv[u] * (face ? wxy2[u] : wxy[u]) + beta * pv[u];
          b[threadIdx.x + u * FT] = v;
          if (own[u] && kk >= k0 && kk < k1) p_new[at[u] + sz * gk] = v;
        }
      if (kk < k1) load(kk + 1);
      __syncthreads();
      const double* m = b + ((ty < t.th ? ty : 0) + 1) * hw + tx + 1;
      const double cc = m[0];
      const double e = (m[-1] + m[1]) + (m[-hw] + m[hw]);
      const double dg = (m[-hw - 1] + m[-hw + 1]) + (m[hw - 1] + m[hw + 1]);
      const double Q = c.w[1] * cc + (c.w[2] * e + c.w[3] * dg);
      if (kk > k0 && in) {
        const int kp = kk - 1;
        double y = P + (Q2 + Q);
        const int faces = faces_xy + on_face(kp, d.nz);
        if (faces) y *= pow2(-faces);
        q[i + sy * j + sz * kp] = y;
        pq += cp * y;
      }
      if (kk >= k0 && kk < k1) P = c.w[0] * cc + (c.w[1] * e + c.w[2] * dg);
      Q2 = Q1;
      Q1 = Q;
      cp = cc;
    }
    __syncthreads();  // the next tile writes the buffers
  }
  pq = block_fold<false, FT>(pq);
  if (threadIdx.x == 0) partial[blockIdx.x] = pq;
  if (!last_block(&s->ticket)) return;
  pq = fold_partials<false, FT>(gridDim.x, partial);
  if (threadIdx.x == 0) {
    s->alpha = s->rz / pq;
    if (!(pq > 0.0)) s->done = 1;
  }
}

// x += alpha p, r -= alpha q, beta = the ratio of the new <r, r/d> to the old.
__global__ void __launch_bounds__(FT) k_cg_update(LevelDev d, HelmCoef c, const double* __restrict__ p,
                                                  const double* __restrict__ q, double* __restrict__ x,
                                                  double* __restrict__ r, double* partial, CgState* s,
                                                  int* host_done) {
  if (s->done) return;
  const double alpha = s->alpha;
  double v2[2] = {0.0, 0.0};  // <r, r>, <r, r/d> d_0
  const long long gs = (long long)gridDim.x * FT;
  auto step = [&](long long n, double xv, double pv, double rv, double qv) {
    int i, j, k;
    node_ijk(d, n, i, j, k);
    x[n] = xv + alpha * pv;
    const double v = rv - alpha * qv;
    r[n] = v;
    v2[0] += v * v;
    v2[1] += v * (v * pow2(on_face(i, d.nx) + on_face(j, d.ny) + on_face(k, d.nz)));
  };
  long long n = blockIdx.x * (long long)FT + threadIdx.x;
  for (; n + gs < d.Nn; n += 2 * gs) {  // two nodes' loads in flight
    const long long m = n + gs;
    const double x0 = x[n], p0 = p[n], r0 = r[n], q0 = q[n];
    const double x1 = x[m], p1 = p[m], r1 = r[m], q1 = q[m];
    step(n, x0, p0, r0, q0);
    step(m, x1, p1, r1, q1);
  }
  if (n < d.Nn) step(n, x[n], p[n], r[n], q[n]);
  block_values<FT>(v2, 2, partial);
  double rr, rz;
  if (!last_block(&s->ticket)) return;
  rr = fold_partials<false, FT>(gridDim.x, partial);
  rz = fold_partials<false, FT>(gridDim.x, partial + gridDim.x) * c.inv_d;
  if (threadIdx.x == 0) {
    s->rr = rr;
    s->beta = rz / s->rz;
    s->rz = rz;
    const int it = s->it + 1, done = rr <= s->tol2 ? 1 : it >= CG_MAX_IT ? 2 : 0;
    s->it = it;
    if (done) *host_done = s->done = done;
  }
}

// gamma~_e = mean of the element's eight nodal values
// (once the solve has converged)
__global__ void k_elem_mean(LevelDev d, const double* __restrict__ x, double* __restrict__ g,
                            const CgState* s) {
  if (s->done != 1) return;
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= d.E) return;
  int i, j, k;
  elem_ijk(d, e, i, j, k);
  const long long sy = d.nx + 1, sz = (long long)(d.nx + 1) * (d.ny + 1);
  const long long n0 = i + sy * (j + (long long)(d.ny + 1) * k);
  double acc = 0.0;
#pragma unroll
  for (int a = 0; a < 8; ++a) acc += x[n0 + (a & 1) + ((a >> 1) & 1) * sy + ((a >> 2) & 1) * sz];
  g[e] = 0.125 * acc;
}

// Tile and march of k_cg_apply.  An FP64 instruction costs a warp the same however few of
// its lanes hold a node, so the tile (16 to 64 wide, as high as 256 threads allow) is
// the one that covers the plane in the fewest blocks: 81 x 81 nodes take 27 tiles of 27
// x 9, 33 of 32 x 8 (67 us an application, 58 now).  A march is as long as leaves the busiest SM
// the least work, zc planes costing zc + 2 with the halo, blocks spread over 152 SMs
// (short marches for small grids, where whole columns would leave SMs idle).
HelmTile helm_tile(const LevelDev& d) {
  HelmTile t = {};
  long long least = 0;
  for (int tw = 16; tw <= 64; ++tw) {
    const int th = FT / tw;
    const long long tx = (d.nx + tw) / tw, ty = (d.ny + th) / th;
    // warps with a node, and the blocks' overhead
    const long long cost = tx * ty * ((tw * th + 31) / 32 * 4 + 1);
    if ((tw + 2) * (th + 2) <= HSLOTS && (!least || cost < least)) {
      least = cost;
      t.tw = tw;
      t.th = th;
      t.tiles_x = (int)tx;
      t.tiles_y = (int)ty;
    }
  }
  const long long tiles = (long long)t.tiles_x * t.tiles_y;
  const int planes = d.nz + 1;
  double cost = 1e300;
  for (int zc = 1; zc <= planes && zc <= 64; ++zc) {
    const long long blocks = tiles * ((planes + zc - 1) / zc);
    const double w = (double)((blocks + 151) / 152) * (zc + 2);
    if (w < cost) {
      cost = w;
      t.zc = zc;
    }
  }
  t.items = tiles * ((planes + t.zc - 1) / t.zc);
  return t;
}

}  // namespace

extern "C" nc_status nc_filter(nc_ctx* ctx, const double* rho, double* gamma_f, double radius,
                               void* stream) {
  if (!ctx || !rho || !gamma_f || !(radius >= 0.0) || !std::isfinite(radius))
    return set_err(ctx, NC_ERR_ARG, "nc_filter: bad argument");
  cudaStream_t s = (cudaStream_t)stream;
  const Level& L = ctx->lv[0];
  const LevelDev& d = L.d;
  const long long Nn = d.Nn;
  nc_status st;
  for (int q = 0; q < 5; ++q)
    if (!ctx->filt[q] &&
        (st = cuda_check(ctx, cudaMalloc((void**)&ctx->filt[q], sizeof(double) * Nn),
                         "cudaMalloc filter")) != NC_OK)
      return st;
  double *x = ctx->filt[0], *r = ctx->filt[1], *q = ctx->filt[2], *p[2] = {ctx->filt[3], ctx->filt[4]};
  const HelmCoef c = helm_coef(d.h, radius);
  CgState* cg = (CgState*)ctx->dscal;
  static_assert(sizeof(CgState) <= sizeof(double) * (MAX_RESTART + 2) * 4, "dscal holds the state");
  cudaGetLastError();  // below, only this call's launches are meant
  cudaMemsetAsync(cg, 0, sizeof(CgState), s);
  const unsigned vb = (unsigned)std::min<long long>((Nn + FT - 1) / FT, RED_BLOCKS_MAX);
  // The end of the solve, which the host looks at while it enqueues: a field that needs few
  // iterations (none, if it is zero) does not pay for the launches of a batch.
  volatile int* const ended = (int*)ctx->pin;
  *ended = 0;
  k_cg_rhs<<<vb, FT, 0, s>>>(d, c, rho, r, x, ctx->partial, cg, (int*)ended);
  const HelmTile tile = helm_tile(d);
  const unsigned ab = (unsigned)std::min<long long>(tile.items, (long long)MAX_RESTART * RED_BLOCKS_MAX);
  CgState h;
  int m = 0, batch = 16;  // a radius of 2.5 h takes about 19 iterations
  do {
    for (int i = 0; i < batch && !*ended; ++i, ++m) {
      k_cg_apply<<<ab, FT, 0, s>>>(d, c, tile, r, p[m & 1], p[(m + 1) & 1], q, ctx->partial, cg);
      k_cg_update<<<vb, FT, 0, s>>>(d, c, p[(m + 1) & 1], q, x, r, ctx->partial, cg, (int*)ended);
    }
    k_elem_mean<<<fblocks(d.E), FT, 0, s>>>(d, x, gamma_f, cg);
    // a refused launch would leave the state, which ends the loop, as it is
    st = cuda_check(ctx, cudaGetLastError(), "nc_filter");
    if (st == NC_OK)
      st = cuda_check(ctx, cudaMemcpyAsync(&h, cg, sizeof(h), cudaMemcpyDeviceToHost, s), "nc_filter");
    // on an error too: no kernel may write to `ended` after the call
    const nc_status done = cuda_check(ctx, cudaStreamSynchronize(s), "nc_filter");
    if (st == NC_OK) st = done;
    if (st != NC_OK) return st;
    // the rest at the rate seen so far
    const double rate = std::log(h.rr / h.bb) / m;
    const double need = rate < 0.0 ? std::log(h.tol2 / h.rr) / rate + 1.0 : 32.0;
    batch = need >= 1.0 && need < 32.0 ? (int)need : 32;
  } while (!h.done);
  if (h.done == 3) return set_err(ctx, NC_ERR_NAN, "nc_filter: non-finite design");
  if (h.done == 2) return set_err(ctx, NC_ERR_MAXIT, "nc_filter: CG did not converge");
  return NC_OK;
}
