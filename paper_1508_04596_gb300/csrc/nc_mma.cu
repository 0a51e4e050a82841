// Design update of the optimisation problem (Sec. 3.2): the volume constraint
// and one iteration of the method of moving asymptotes (MMA, Svanberg 1987)
// for one inequality constraint.
//
// MMA as implemented (the paper names the method and prints no details):
//  * asymptotes: iterations 0 and 1 put L, U at x -/+ 0.5 (xmax - xmin); later
//    ones widen them by 1.2 where a variable moved the same way twice, narrow
//    them by 0.7 where it oscillated, and keep them within 0.01 .. 10 times
//    (xmax - xmin) of x;
//  * move limits: alpha = max(xmin, L + 0.1 (x - L), x - move d),
//    beta = min(xmax, U - 0.1 (U - x), x + move d), d = xmax - xmin;
//  * each function f_i (objective, constraint) is replaced by the separable
//    convex approximation with p = (U - x)^2 (1.001 a+ + 0.001 a- + 1e-5 / d),
//    q = (x - L)^2 (0.001 a+ + 1.001 a- + 1e-5 / d), a = df_i/dx_j;
//  * the subproblem is solved through its dual: for a multiplier lam the
//    minimiser of the Lagrangian is, per variable, the clipped
//    (L sqrt(P) + U sqrt(Q)) / (sqrt(P) + sqrt(Q)), P = p0 + lam p1,
//    Q = q0 + lam q1, and the approximated constraint does not increase with
//    lam; lam = 0 if it already holds, else lam is bracketed from 1 upwards and
//    the bracket closed by inverse quadratic interpolation safeguarded by
//    bisection (Chandrupatla 1997) until it is a few units in the last place
//    wide; lam is the end at which the approximated constraint holds.
//
// The search runs on the device.  Every evaluation of the approximated constraint
// is one pass over the variables (fixed-partition reduction, deterministic); the
// block that finishes a pass last folds the partial sums in index order and one
// thread takes the next step of the search, whose state stays in device memory.
// The host enqueues a batch of passes, waits and finds what the last of them wrote to
// page-locked memory: passes after the search has ended return at once.  Measured at 80x80x160 (1.02M variables, 432k
// active): 57 bisection passes of 117 us, each followed by a host read, took 8.1 ms
// for the volume and the update.  10-15 passes are needed now, and each takes the
// coefficients of the active variables, computed once per call, from a compacted
// workspace.  A pass is bound by the FP64 pipe (71 % busy on an SM that works, 41 % over the pass:
// the active variables lie unevenly over the blocks); for a variable inside its limits
//   p1/(U - y) + q1/(y - L) = (sqrt P + sqrt Q) (p1/sqrt P + q1/sqrt Q) / (U - L),
// and at a limit the term does not depend on lam, so a pass takes two reciprocal
// square roots per variable and no division: 49 us a pass, 0.92 ms for the volume
// and the update (73 us and 1.22 ms with two square roots and two divisions).
#include <cmath>

#include "nc_internal.cuh"
#include "nc_reduce.cuh"

namespace nc {
nc_status set_err(nc_ctx* ctx, nc_status st, const std::string& msg);
nc_status cuda_check(nc_ctx* ctx, cudaError_t e, const char* what);
}  // namespace nc

using namespace nc;

namespace {

constexpr int MT = 256;
// Passes enqueued between two reads of the search's state: the search takes 10-15
// evaluations, and one that finds it ended costs about 2 us.  Where the constraint holds
// without a multiplier there is nothing to search for: the host reads what the first
// evaluation found while MMA_FIRST passes keep the GPU busy, and only then enqueues the rest.
constexpr int MMA_FIRST = 2, MMA_BATCH = 14;

// Blocks of a reduction over n variables: four per SM at most (FP64 square roots and
// divisions are long dependent chains), a partition that depends only on n.
inline unsigned mma_blocks(long long n) {
  const long long b = (n + MT - 1) / MT;
  return (unsigned)(b < RED_BLOCKS_MAX ? b : RED_BLOCKS_MAX);
}

// Block sum (or maximum) of one value per thread -> partial[blockIdx.x].
template <bool MAX>
__device__ __forceinline__ void block_partial(double v, double* partial) {
  v = block_fold<MAX, MT>(v);
  if (threadIdx.x == 0) partial[blockIdx.x] = v;
}

// out[0], out[1]: sums of (1 - gamma_e) and of the active count over the variables; the same to
// page-locked memory
__global__ void __launch_bounds__(MT) k_volume(long long n, const double* __restrict__ g,
                                               const unsigned char* __restrict__ active,
                                               double* partial, double* out, double* host, unsigned* ticket) {
  double acc = 0.0, cnt = 0.0;
  for (long long j = blockIdx.x * (long long)MT + threadIdx.x; j < n; j += (long long)gridDim.x * MT) {
    if (active && !active[j]) continue;
    acc += 1.0 - g[j];
    cnt += 1.0;
  }
  block_partial<false>(acc, partial);
  block_partial<false>(cnt, partial + gridDim.x);
  if (!last_block(ticket)) return;
  const double s0 = fold_partials<false, MT>(gridDim.x, partial);
  const double s1 = fold_partials<false, MT>(gridDim.x, partial + gridDim.x);
  if (threadIdx.x == 0) {
    out[0] = host[0] = s0;
    out[1] = host[1] = s1;
  }
}

// dg = -1/(vf count) on active entries, 0 elsewhere; nothing without an active one
__global__ void k_volume_grad(long long n, const unsigned char* __restrict__ active,
                              const double* __restrict__ sums, double vf, double* __restrict__ dg) {
  __shared__ double sh;
  if (threadIdx.x == 0) sh = -(1.0 / (vf * sums[1]));  // one FP64 division per block
  __syncthreads();
  const double dgval = sh;
  const long long j = blockIdx.x * (long long)MT + threadIdx.x;
  if (j >= n || !(sums[1] > 0.0)) return;
  dg[j] = (!active || active[j]) ? dgval : 0.0;
}

// Asymptotes of iteration k of one variable, in place.
__device__ __forceinline__ void mma_asym(long long j, int k, double xj,
                                         const double* __restrict__ xo1,
                                         const double* __restrict__ xo2, double* low, double* upp,
                                         double xmin, double xmax) {
  const double d = xmax - xmin;
  if (k < 2) {
    low[j] = xj - 0.5 * d;
    upp[j] = xj + 0.5 * d;
    return;
  }
  const double o1 = xo1[j];
  const double s = (xj - o1) * (o1 - xo2[j]);
  const double fac = s < 0.0 ? 0.7 : (s > 0.0 ? 1.2 : 1.0);
  double l = xj - fac * (o1 - low[j]);
  double u = xj + fac * (upp[j] - o1);
  l = fmin(fmax(l, xj - 10.0 * d), xj - 0.01 * d);
  u = fmin(fmax(u, xj + 0.01 * d), xj + 10.0 * d);
  low[j] = l;
  upp[j] = u;
}

// What the separable Lagrangian of one variable needs for any multiplier.  w =
// 1/(u - l); c, ta, tb: the variable's term p1/(u - y) + q1/(y - l) of the
// approximated constraint at y = x, and at alpha and beta less c.
struct MmaCoef {
  double l, u, alpha, beta, p0, q0, p1, q1, w, c, ta, tb;
};
constexpr int MMA_COEFS = 12;

// The arithmetic from here to mma_term names its rounded products and fuses only where it says
// so (the evaluations, which the FP64 pipe bounds): left to the compiler, kernels that read the
// coefficients and kernels that form them fuse different operations, and the design would
// depend on which of them ran.
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }

// The coefficients but for w, c, ta and tb, which only the evaluations need.
__device__ __forceinline__ MmaCoef mma_coef_y(double xj, double l, double u, double a0, double a1,
                                              double xmin, double xmax, double move, double r) {
  const double d = xmax - xmin;
  const double a0p = fmax(a0, 0.0), a0m = fmax(-a0, 0.0);
  const double a1p = fmax(a1, 0.0), a1m = fmax(-a1, 0.0);
  const double ux = u - xj, xl = xj - l, ux2 = mul(ux, ux), xl2 = mul(xl, xl);
  MmaCoef m;
  m.l = l;
  m.u = u;
  m.p0 = mul(ux2, mul(1.001, a0p) + mul(0.001, a0m) + r);
  m.q0 = mul(xl2, mul(0.001, a0p) + mul(1.001, a0m) + r);
  m.p1 = mul(ux2, mul(1.001, a1p) + mul(0.001, a1m) + r);
  m.q1 = mul(xl2, mul(0.001, a1p) + mul(1.001, a1m) + r);
  m.alpha = fmax(fmax(xmin, l + mul(0.1, xl)), xj - mul(move, d));
  m.beta = fmin(fmin(xmax, u - mul(0.1, ux)), xj + mul(move, d));
  m.alpha = fmin(m.alpha, m.beta);  // limits that cross (x far outside the box): the upper one holds
  return m;
}

__device__ __forceinline__ double mma_term_at(const MmaCoef& m, double y) {
  const double a = m.u - y, b = y - m.l;
  return fma(m.p1, b, mul(m.q1, a)) / mul(a, b);
}

__device__ __forceinline__ MmaCoef mma_coef(double xj, double l, double u, double a0, double a1,
                                            double xmin, double xmax, double move, double r) {
  MmaCoef m = mma_coef_y(xj, l, u, a0, a1, xmin, xmax, move, r);
  m.w = 1.0 / (u - l);
  m.c = mma_term_at(m, xj);
  m.ta = mma_term_at(m, m.alpha) - m.c;
  m.tb = mma_term_at(m, m.beta) - m.c;
  return m;
}

// Minimiser y_j(lam) of the separable Lagrangian, clipped to [alpha, beta].
__device__ __forceinline__ double mma_y(const MmaCoef& m, double lam) {
  const double sP = sqrt(m.p0 + mul(lam, m.p1)), sQ = sqrt(m.q0 + mul(lam, m.q1));
  return fmin(fmax((mul(m.l, sP) + mul(m.u, sQ)) / (sP + sQ), m.alpha), m.beta);
}
// Its term of the approximated constraint (P, Q > 0: the approximation adds 1e-5 / d).
// Where P or Q is infinite (an infinite entry of df0), y is not a number and mma_y gives
// alpha; the first comparison below is written so that the term goes with it.
__device__ __forceinline__ double mma_term(const MmaCoef& m, double lam) {
  const double P = fma(lam, m.p1, m.p0), Q = fma(lam, m.q1, m.q0);
  const double rP = rsqrt(P), rQ = rsqrt(Q), sP = mul(P, rP), sQ = mul(Q, rQ);
  const double den = sP + sQ, num = fma(m.l, sP, mul(m.u, sQ));  // y = num / den
  const double t = fma(mul(den, m.w), fma(m.p1, rP, mul(m.q1, rQ)), -m.c);
  return !(num > mul(m.alpha, den)) ? m.ta : (num >= mul(m.beta, den) ? m.tb : t);
}

// The search for the multiplier.  a is the newest point, b the end of the bracket
// on the other side of the root, c the point before (phase 2); while bracketing
// (phase 1) b is the largest multiplier known to violate the constraint.
struct MmaSearch {
  double lam, a, fa, b, fb, c, fc, change;
  int phase, evals, done, err;
  unsigned ticket, pad;
};

// One step of the search: v = f(s.lam) = f1 + sum.
__device__ void mma_advance(MmaSearch& s, double f1, double sum) {
  const double v = f1 + sum;
  ++s.evals;
  if (!isfinite(sum)) {
    s.err = s.done = 1;
    return;
  }
  constexpr double LAM_MAX = 1.6069380442589903e60;  // 2^200
  double t;
  if (s.phase == 0) {  // v = f(0)
    if (v <= 0.0) {
      s.done = 1;
      return;
    }
    s.b = 0.0;
    s.fb = v;
    s.lam = 1.0;
    s.phase = 1;
    return;
  }
  if (s.phase == 1) {
    if (v > 0.0) {
      if (s.lam >= 0.5 * LAM_MAX) {  // no multiplier satisfies it
        s.lam = LAM_MAX;
        s.done = 1;
        return;
      }
      s.b = s.lam;
      s.fb = v;
      s.lam = fmin(s.lam * (s.evals < 4 ? 2.0 : 16.0), 0.5 * LAM_MAX);
      return;
    }
    s.a = s.lam;
    s.fa = v;
    s.c = s.b;
    s.fc = s.fb;
    t = fmin(fmax(s.fa / (s.fa - s.fb), 1e-3), 1.0 - 1e-3);  // secant
    s.phase = 2;
  } else {
    if ((v > 0.0) == (s.fa > 0.0)) {
      s.c = s.a;
      s.fc = s.fa;
    } else {
      s.c = s.b;
      s.fc = s.fb;
      s.b = s.a;
      s.fb = s.fa;
    }
    s.a = s.lam;
    s.fa = v;
    const double w = fabs(s.b - s.a), big = fmax(s.a, s.b), small = fmin(s.a, s.b);
    const double tol = 4.4e-16 * big;
    if (w <= 2.0 * tol || s.evals >= 400) {
      s.lam = s.fa <= 0.0 ? s.a : s.b;
      s.done = 1;
      return;
    }
    t = 0.5;
    const double xi = (s.a - s.b) / (s.c - s.b), ph = (s.fa - s.fb) / (s.fc - s.fb);
    if (s.fc != s.fa && s.fc != s.fb && ph * ph < xi && (1.0 - ph) * (1.0 - ph) < 1.0 - xi)
      t = s.fa / (s.fb - s.fa) * s.fc / (s.fb - s.fc) +
          (s.c - s.a) / (s.b - s.a) * s.fa / (s.fc - s.fa) * s.fb / (s.fc - s.fb);
    else if (small > 0.0 && big > 4.0 * small)
      t = (sqrt(s.a * s.b) - s.a) / (s.b - s.a);  // bisect the exponent of a wide bracket
    else if (small == 0.0)
      t = (big * (1.0 / 64) - s.a) / (s.b - s.a);
    const double tl = tol / w;
    t = fmin(fmax(t, tl), 1.0 - tl);
  }
  s.lam = s.a + t * (s.b - s.a);
}

// Variables are taken in tiles of MT entries, tile b + i * gridDim.x by block b.
// With a workspace a block stores its active variables' coefficients one after the
// other in its own segment (seg entries), in tile order: slot(first) of a tile is
// the block's running count of active variables.
struct MmaWs {
  double* v;        // MMA_COEFS arrays of gridDim.x * seg entries
  int* cnt;         // active variables per block
  long long seg;    // tiles per block * MT
};

// position of this thread's variable among the block's active ones of this tile,
// and their number (every thread of the block calls it)
__device__ __forceinline__ int tile_slot(bool act, int& total) {
  __shared__ int wc[MT / 32];
  const unsigned m = __ballot_sync(0xffffffffu, act);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) wc[wid] = __popc(m);
  __syncthreads();
  int pos = __popc(m & ((1u << lane) - 1u));
  total = 0;
#pragma unroll
  for (int w = 0; w < MT / 32; ++w) {
    if (w < wid) pos += wc[w];
    total += wc[w];
  }
  return pos;
}

// entry i of the workspace; EVAL: what an evaluation takes, else what y takes
template <bool EVAL>
__device__ __forceinline__ MmaCoef ws_load(const MmaWs& w, long long i) {
  const long long st = (long long)gridDim.x * w.seg;
  MmaCoef m;
  m.l = w.v[i];
  m.u = w.v[i + st];
  m.alpha = w.v[i + 2 * st];
  m.beta = w.v[i + 3 * st];
  m.p0 = w.v[i + 4 * st];
  m.q0 = w.v[i + 5 * st];
  m.p1 = w.v[i + 6 * st];
  m.q1 = w.v[i + 7 * st];
  if (EVAL) {
    m.w = w.v[i + 8 * st];
    m.c = w.v[i + 9 * st];
    m.ta = w.v[i + 10 * st];
    m.tb = w.v[i + 11 * st];
  }
  return m;
}

// The last block's part of an evaluation pass: fold the partials, step the search; its end
// (lam, err, done) goes to page-locked memory too.
__device__ __forceinline__ void mma_finish(double acc, double f1, double* partial, MmaSearch* s, MmaSearch* host) {
  block_partial<false>(acc, partial);
  if (!last_block(&s->ticket)) return;
  const double sum = fold_partials<false, MT>(gridDim.x, partial);
  if (threadIdx.x == 0) {
    MmaSearch t = *s;
    mma_advance(t, f1, sum);
    *s = t;
    if (t.done) {
      host->lam = t.lam;
      host->err = t.err;
      host->done = t.done;
    }
  }
}

struct MmaArgs {
  long long n;
  const double *x, *xo1, *xo2, *df0, *df1;
  double *low, *upp;
  const unsigned char* active;
  double xmin, xmax, move, r, scale0, f1;  // r = 1e-5 / (xmax - xmin)
};

// Asymptotes of the iteration, the coefficients into the workspace (STORE), and the
// first evaluation, at lam = 0.
template <bool STORE>
__global__ void __launch_bounds__(MT) k_mma_begin(MmaArgs a, int iter, MmaWs w, double* partial,
                                                  MmaSearch* s, MmaSearch* host) {
  double acc = 0.0;
  const long long base = (long long)blockIdx.x * w.seg;
  long long cnt = 0;
  for (long long j0 = blockIdx.x * (long long)MT; j0 < a.n; j0 += (long long)gridDim.x * MT) {
    const long long j = j0 + threadIdx.x;
    const bool act = j < a.n && (!a.active || a.active[j]);
    int total = 0, pos = 0;
    if (STORE) pos = tile_slot(act, total);
    if (act) {
      const double xj = a.x[j];
      mma_asym(j, iter, xj, a.xo1, a.xo2, a.low, a.upp, a.xmin, a.xmax);
      const MmaCoef m = mma_coef(xj, a.low[j], a.upp[j], a.scale0 * a.df0[j], a.df1[j], a.xmin,
                                 a.xmax, a.move, a.r);
      acc += mma_term(m, 0.0);
      if (STORE) {
        const double q[MMA_COEFS] = {m.l, m.u, m.alpha, m.beta, m.p0, m.q0,
                                     m.p1, m.q1, m.w, m.c, m.ta, m.tb};
#pragma unroll
        for (int r = 0; r < MMA_COEFS; ++r)
          w.v[r * (long long)gridDim.x * w.seg + base + cnt + pos] = q[r];
      }
    }
    cnt += total;
  }
  if (STORE && threadIdx.x == 0) w.cnt[blockIdx.x] = (int)cnt;
  mma_finish(acc, a.f1, partial, s, host);
}

// One evaluation of the approximated constraint at the search's multiplier, with the same
// bits whether the coefficients come from the workspace (STORE) or from the variables.  Three
// blocks per SM: at two (92 registers) 110,592 variables take a second wave, 950 us instead of
// 855 for an update of about 50 passes.
template <bool STORE>
__global__ void __launch_bounds__(MT, 3) k_mma_dual(MmaArgs a, MmaWs w, double* partial, MmaSearch* s,
                                                 MmaSearch* host) {
  if (s->done) return;
  const double lam = s->lam;
  double acc = 0.0;
  if (STORE) {
    const int cnt = w.cnt[blockIdx.x];
    const long long base = (long long)blockIdx.x * w.seg;
    for (int i = threadIdx.x; i < cnt; i += MT) acc += mma_term(ws_load<true>(w, base + i), lam);
  } else {
    // the same sums in the same order: a term goes to the thread that would read its entry
    __shared__ double term[MT];
    int at = 0;  // active variables of the block so far, modulo MT
    for (long long j0 = blockIdx.x * (long long)MT; j0 < a.n; j0 += (long long)gridDim.x * MT) {
      const long long j = j0 + threadIdx.x;
      const bool act = j < a.n && (!a.active || a.active[j]);
      int total;
      const int pos = tile_slot(act, total);
      if (act)
        term[(at + pos) % MT] = mma_term(mma_coef(a.x[j], a.low[j], a.upp[j], a.scale0 * a.df0[j], a.df1[j],
                                                  a.xmin, a.xmax, a.move, a.r), lam);
      __syncthreads();
      if ((int)(threadIdx.x + MT - at) % MT < total) acc += term[threadIdx.x];
      at = (at + total) % MT;
    }
  }
  mma_finish(acc, a.f1, partial, s, host);
}

// x^{k+1} = y(lam) once the search has ended; the previous iterates shift;
// host->change = max |y - x|.
template <bool STORE>
__global__ void __launch_bounds__(MT) k_mma_commit(MmaArgs a, MmaWs w, double* x, double* xo1,
                                                   double* xo2, double* partial, MmaSearch* s,
                                                   MmaSearch* host) {
  if (!s->done || s->err) return;
  const double lam = s->lam;
  double mx = 0.0;
  long long at = (long long)blockIdx.x * w.seg;
  for (long long j0 = blockIdx.x * (long long)MT; j0 < a.n; j0 += (long long)gridDim.x * MT) {
    const long long j = j0 + threadIdx.x;
    const bool act = j < a.n && (!a.active || a.active[j]);
    int total = 0, pos = 0;
    if (STORE) pos = tile_slot(act, total);
    if (j < a.n) {
      const double xj = x[j];
      double y = xj;
      if (act)
        y = mma_y(STORE ? ws_load<false>(w, at + pos)
                        : mma_coef_y(xj, a.low[j], a.upp[j], a.scale0 * a.df0[j], a.df1[j], a.xmin,
                                     a.xmax, a.move, a.r), lam);
      xo2[j] = xo1[j];
      xo1[j] = xj;
      x[j] = y;
      mx = fmax(mx, fabs(y - xj));
    }
    at += total;
  }
  block_partial<true>(mx, partial);
  if (!last_block(&s->ticket)) return;
  const double v = fold_partials<true, MT>(gridDim.x, partial);
  if (threadIdx.x == 0) host->change = v;
}

// out = clamp(in, lo, hi) on active entries, fixed (or 0) elsewhere
__global__ void k_design_map(long long n, const double* in, const unsigned char* __restrict__ active,
                             const double* __restrict__ fixed, double lo, double hi, double* out) {
  const long long j = blockIdx.x * (long long)MT + threadIdx.x;
  if (j >= n) return;
  if (!active || active[j])
    out[j] = fmin(fmax(in[j], lo), hi);
  else
    out[j] = fixed ? fixed[j] : 0.0;
}

inline unsigned grid1(long long n) { return (unsigned)((n + MT - 1) / MT); }

// The coefficient workspace of nc_mma_update, kept by the context (grown when a
// larger problem asks).  False if the device would keep less than 8 GB free: the
// passes then recompute the coefficients from the variables.
bool mma_workspace(nc_ctx* ctx, long long n, unsigned nb, MmaWs& w) {
  const long long tiles = (n + MT - 1) / MT;
  w.seg = (tiles + nb - 1) / nb * MT;
  w.v = nullptr;
  w.cnt = nullptr;
  if (w.seg > 0x7fffffffLL) return false;
  const size_t vals = (size_t)MMA_COEFS * nb * w.seg, need = sizeof(double) * vals + sizeof(int) * nb;
  if (ctx->mma_ws_bytes < need) {
    size_t fr = 0, tot = 0;
    if (cudaMemGetInfo(&fr, &tot) != cudaSuccess || fr < need + ((size_t)8 << 30)) {
      cudaGetLastError();
      return false;
    }
    void* p = nullptr;
    if (cudaMalloc(&p, need) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    cudaFree(ctx->mma_ws);
    ctx->mma_ws = p;
    ctx->mma_ws_bytes = need;
  }
  w.v = (double*)ctx->mma_ws;
  w.cnt = (int*)(w.v + vals);
  return true;
}

}  // namespace

extern "C" {

void nc_default_mma_opts(nc_mma_opts* o) {
  if (!o) return;
  o->move = 0.2;
  o->xmin = 0.0;
  o->xmax = 1.0;
  o->df0_scale = 1.0;
}

nc_status nc_design_map(nc_ctx* ctx, long long n, const double* in, const unsigned char* active,
                        const double* fixed, double lo, double hi, double* out, void* stream) {
  if (!ctx) return NC_ERR_ARG;
  if (!in || !out || n < 1 || !(hi >= lo))
    return set_err(ctx, NC_ERR_ARG, "nc_design_map: invalid argument");
  k_design_map<<<grid1(n), MT, 0, (cudaStream_t)stream>>>(n, in, active, fixed, lo, hi, out);
  return cuda_check(ctx, cudaGetLastError(), "nc_design_map");
}

nc_status nc_volume(nc_ctx* ctx, long long n, const double* gamma, const unsigned char* active,
                    double vf, double* g_host, double* dgdgamma, void* stream) {
  if (!ctx) return NC_ERR_ARG;
  if (!gamma || !g_host || n < 1 || !(vf > 0.0))
    return set_err(ctx, NC_ERR_ARG, "nc_volume: invalid argument");
  cudaStream_t s = (cudaStream_t)stream;
  unsigned* ticket = (unsigned*)(ctx->dscal + 2);
  cudaMemsetAsync(ticket, 0, sizeof(unsigned), s);
  double* const sc = (double*)ctx->pin;
  k_volume<<<mma_blocks(n), MT, 0, s>>>(n, gamma, active, ctx->partial, ctx->dscal, sc, ticket);
  // the host waits for the sums alone; the gradient is left on the stream
  nc_status st = cuda_check(ctx, cudaEventRecord(ctx->ev, s), "nc_volume");
  if (dgdgamma) k_volume_grad<<<grid1(n), MT, 0, s>>>(n, active, ctx->dscal, vf, dgdgamma);
  if (st == NC_OK) st = cuda_check(ctx, cudaEventSynchronize(ctx->ev), "nc_volume");
  if (st == NC_OK) st = cuda_check(ctx, cudaGetLastError(), "nc_volume");
  if (st != NC_OK) return st;
  if (!(sc[1] > 0.0)) return set_err(ctx, NC_ERR_ARG, "nc_volume: no active variable");
  *g_host = sc[0] * (1.0 / (vf * sc[1])) - 1.0;
  return NC_OK;
}

nc_status nc_mma_update(nc_ctx* ctx, long long n, int iter, double* x, double* xold1,
                        double* xold2, double* low, double* upp, const double* df0, double f1,
                        const double* df1, const unsigned char* active, const nc_mma_opts* opts,
                        double* lambda_host, double* change_host, void* stream) {
  if (!ctx) return NC_ERR_ARG;
  nc_mma_opts o;
  nc_default_mma_opts(&o);
  if (opts) o = *opts;
  if (!x || !xold1 || !xold2 || !low || !upp || !df0 || !df1 || n < 1 || iter < 0 ||
      !(o.xmax > o.xmin) || !(o.move > 0.0) || !std::isfinite(f1) || !(o.df0_scale > 0.0))
    return set_err(ctx, NC_ERR_ARG, "nc_mma_update: invalid argument");
  cudaStream_t s = (cudaStream_t)stream;
  const unsigned nb = mma_blocks(n);
  MmaWs w;
  const bool store = mma_workspace(ctx, n, nb, w);
  const MmaArgs a{n, x, xold1, xold2, df0, df1, low, upp, active, o.xmin, o.xmax, o.move,
                  1e-5 / (o.xmax - o.xmin), o.df0_scale, f1};
  MmaSearch* srch = (MmaSearch*)ctx->dscal;
  static_assert(sizeof(MmaSearch) <= sizeof(double) * (MAX_RESTART + 2) * 4, "dscal holds the search");
  cudaGetLastError();  // below, only this call's launches are meant
  cudaMemsetAsync(srch, 0, sizeof(MmaSearch), s);
  double* part = ctx->partial;
  // the end of the search and the change, written by the kernels: a copy between the first
  // evaluation and the next would cost a small update 4 to 8 %
  MmaSearch* const h = (MmaSearch*)ctx->pin;
  static_assert(sizeof(MmaSearch) <= PIN_BYTES, "ctx->pin holds the search");
  *h = MmaSearch{};
  if (store)
    k_mma_begin<true><<<nb, MT, 0, s>>>(a, iter, w, part, srch, h);
  else
    k_mma_begin<false><<<nb, MT, 0, s>>>(a, iter, w, part, srch, h);
  auto search = [&](int passes) {
    for (int i = 0; i < passes; ++i) {
      if (store)
        k_mma_dual<true><<<nb, MT, 0, s>>>(a, w, part, srch, h);
      else
        k_mma_dual<false><<<nb, MT, 0, s>>>(a, w, part, srch, h);
    }
  };
  nc_status st = cuda_check(ctx, cudaEventRecord(ctx->ev, s), "nc_mma_update");
  search(MMA_FIRST);
  if (st == NC_OK) st = cuda_check(ctx, cudaEventSynchronize(ctx->ev), "nc_mma_update");
  int passes = h->done ? 0 : MMA_BATCH;
  do {  // most searches end within the first batch; a pass after the end costs its launch
    if (st == NC_OK) {
      search(passes);
      passes = MMA_BATCH;
      if (store)
        k_mma_commit<true><<<nb, MT, 0, s>>>(a, w, x, xold1, xold2, part, srch, h);
      else
        k_mma_commit<false><<<nb, MT, 0, s>>>(a, w, x, xold1, xold2, part, srch, h);
      // a refused launch would leave the state, which ends the loop, as it is
      st = cuda_check(ctx, cudaGetLastError(), "nc_mma_update");
    }
    // on an error too: no pass may write to h after the call
    const nc_status done = cuda_check(ctx, cudaStreamSynchronize(s), "nc_mma_update");
    if (st == NC_OK) st = done;
    if (st != NC_OK) return st;
  } while (!h->done);
  if (h->err) return set_err(ctx, NC_ERR_NAN, "nc_mma_update: non-finite value");
  if (lambda_host) *lambda_host = h->lam;
  if (change_host) *change_host = h->change;
  return NC_OK;
}

}  // extern "C"
