// Element operators by warps that march along y.
//
// A lane owns an x-node face: the nodes (i, j..j+1, k..k+1) of one element layer k.
// The faces of a layer stack, numbered l = i + (nx + 1) k, are cut into chunks of 31
// (32 where no element would straddle two chunks), a warp per chunk; lane L's element
// lies between its own face and lane L + 1's, and the last lane of a chunk only
// receives.  A warp marches over up to rc element rows j.  What neighbouring elements
// share is then formed once:
//  * z stage of the interpolation: once per vertical grid edge (the row above becomes
//    the row below of the next step), instead of by the four elements around it;
//  * y stage: once per face, handed to the left element by a shuffle;
//  * the transposed stages mirror this: a face's two elements are added by a shuffle
//    before or after the y stage, the rows of two steps are added in registers, and
//    the z stage runs on the sums.
// A step then loads 2 nodes per lane and vector (8 with a thread per element) and
// writes 10 sums (40), and the gather adds the two element layers of a node (40 rows).
// Loads of the next row are in flight (cp.async into the warp's own shared memory, so
// they hold no registers) while a step computes.  At 192x192x384 the FP32 J v takes
// 0.99 ms and its gather 0.27 (1.28 and 0.42 with a thread and 40 rows per element),
// at 96^3 84 us together (119), J^T w 88 (119); FP64 J v from the store at 96^3 2.03 ms
// (2.35), the residual 1.80 (2.08).
//
// FP32 products act on pairs: (state, direction) in the z and y stages, the two Gauss
// points of a pair along x in the fluxes, and the two faces in the transposed y
// stage.  They are bound by latency at two warps per scheduler (255 registers; three,
// with spills, are 30 % slower).  FP64 kernels are bound by their FP64 instruction count
// (a warp instruction takes a scheduler's FP64 unit 64 cycles), so they sum the two
// faces first and select with integer moves.
//
// A lane whose face ends a row of elements (i = nx) or a chunk has no element: it
// shuffles with itself, so its arithmetic sees only values of its own face, and its
// results are dropped (FP64) or weighted by zero (FP32).  A non-finite value thus
// reaches no rows but those of its own elements.
#pragma once
#include "nc_element_f2.cuh"
#include "nc_internal.cuh"

namespace nc {
namespace march {

enum Kind { RES, JVP, JTVP, SENS, LINEARIZE, JVP_LIN, JTVP_LIN };

constexpr int WARPS = 4;     // warps per block at most
constexpr int ROWS = 10;     // sums per face and node row: 5 fields at both z corners
constexpr int ROW_LEN = ROWS * 32;

// ---------------------------------------------------------------- pairs
struct d2 {
  double x, y;
};
template <typename R> struct PairOf;
template <> struct PairOf<float> { typedef f2 T; };
template <> struct PairOf<double> { typedef d2 T; };
template <typename R> using PR = typename PairOf<R>::T;

__device__ __forceinline__ f2 mk(float a, float b) { return mk2(a, b); }
__device__ __forceinline__ d2 mk(double a, double b) { return d2{a, b}; }
__device__ __forceinline__ f2 vadd(f2 a, f2 b) { return add2(a, b); }
__device__ __forceinline__ d2 vadd(d2 a, d2 b) { return d2{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ float vadd(float a, float b) { return a + b; }
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ f2 vsub(f2 a, f2 b) { return sub2(a, b); }
__device__ __forceinline__ d2 vsub(d2 a, d2 b) { return d2{a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ float vsub(float a, float b) { return a - b; }
__device__ __forceinline__ double vsub(double a, double b) { return a - b; }
// c a + b
__device__ __forceinline__ f2 vfma(float c, f2 a, f2 b) { return fma2(bc2(c), a, b); }
__device__ __forceinline__ d2 vfma(double c, d2 a, d2 b) { return d2{fma(c, a.x, b.x), fma(c, a.y, b.y)}; }
__device__ __forceinline__ float vfma(float c, float a, float b) { return fmaf(c, a, b); }
__device__ __forceinline__ double vfma(double c, double a, double b) { return fma(c, a, b); }

template <typename R> __device__ __forceinline__ R shfl1(R v, int src) {
  return __shfl_sync(0xffffffffu, v, src);
}
__device__ __forceinline__ float shfl(float v, int s) { return shfl1(v, s); }
__device__ __forceinline__ double shfl(double v, int s) { return shfl1(v, s); }
__device__ __forceinline__ f2 shfl(f2 v, int s) { return mk(shfl1(v.x, s), shfl1(v.y, s)); }
__device__ __forceinline__ d2 shfl(d2 v, int s) { return mk(shfl1(v.x, s), shfl1(v.y, s)); }

// component s of an interpolated quantity: 0 the state, 1 the direction
template <int s> __device__ __forceinline__ float comp(f2 v) { return s ? v.y : v.x; }
template <int s> __device__ __forceinline__ double comp(d2 v) { return s ? v.y : v.x; }
template <int s> __device__ __forceinline__ float comp(float v) { return v; }
template <int s> __device__ __forceinline__ double comp(double v) { return v; }

template <typename R>
__device__ __forceinline__ void copy_async(R* dst, const R* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if (sizeof(R) == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_wait() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// What a kind interpolates: both vectors (pairs), the state alone or the direction
// alone; VEL: it also reads the state's velocities (products from the store).
template <int K> struct Traits {
  static constexpr bool TWO = K == JVP || K == JTVP || K == SENS;
  static constexpr bool DIR = K == JVP_LIN || K == JTVP_LIN;  // the direction alone
  static constexpr bool VEL = DIR;
  static constexpr bool TEST = K != SENS && K != LINEARIZE;
  static constexpr bool ADJ = K == JTVP || K == JTVP_LIN;
};

// z stage of one vertical edge: the difference and the values at both Gauss planes.
template <typename T> struct Edge {
  T dz, v[2];
};

// Per-warp staging of one node row: [field * 2 + z][lane], and the state's velocities.
template <typename R, int K> struct Stage {
  typedef typename std::conditional<Traits<K>::TWO, PR<R>, R>::type T;
  T n[10][32];
  R u[Traits<K>::VEL ? 6 : 1][Traits<K>::VEL ? 32 : 1];
};

template <typename R, int K>
__global__ void __launch_bounds__(WARPS * 32, 2) k_march(LevelDev d, ElemConst<R> c, MarchPlan mp,
                                                        const R* __restrict__ x_,
                                                        const R* __restrict__ gam,
                                                        const R* __restrict__ srcs,
                                                        const R* cache_,
                                                        const R* __restrict__ v_, R* out) {
  chained();
  const R* const x = fresh(x_);
  const R* const cache = fresh(cache_);
  const R* const v = fresh(v_);
  typedef Traits<K> TR;
  typedef typename Stage<R, K>::T T;
  typedef PR<R> P;
  constexpr bool PACKED = std::is_same<R, float>::value && TR::TWO;
  // the row below, the row above and the next one; the row below stays staged only
  // where its velocities are read again (the adjoint)
  constexpr int BUFS = TR::ADJ ? 3 : 2;
  __shared__ Stage<R, K> stage[WARPS][BUFS];
  const int lane = threadIdx.x & 31;
  const long long w = blockIdx.x * (long long)(blockDim.x >> 5) + (threadIdx.x >> 5);
  if (w >= mp.warps()) return;
  const int run = mp.flat ? 0 : (int)(w / mp.nchunk);
  const long long chunk = w - run * mp.nchunk;

  // ---- this lane's face
  const long long faces = (long long)(d.nx + 1) * d.nz * (mp.flat ? d.ny : 1);
  const long long l = min(chunk * mp.stride + lane, faces - 1);
  const bool valid = chunk * mp.stride + lane < faces;
  int i, k, j0;
  split3(l, faces, d.nx + 1, d.nz, i, k, j0);
  if (!mp.flat) j0 = run * mp.rc;
  const int rows = mp.flat ? 1 : min(mp.rc, d.ny - j0);
  const bool elem = valid && lane < 31 && i < d.nx;  // the element to the right is this lane's
  const bool left = valid && lane > 0 && i > 0;      // lane - 1 has the element to the left
  const int to_right = elem ? lane + 1 : lane, to_left = left ? lane - 1 : lane;
  const R mleft = left ? R(1) : R(0);

  const long long sx = d.nx + 1, sxy = sx * (d.ny + 1);
  long long n = i + sx * (j0 + (long long)(d.ny + 1) * k);
  long long e = min(i, d.nx - 1) + (long long)d.nx * (j0 + (long long)d.ny * k);
  Stage<R, K>* const sh = stage[threadIdx.x >> 5];
  uint8_t fl0[2] = {0, 0}, fl[2] = {0, 0};  // Dirichlet flags of the first and of the next row

  auto issue = [&](int b, long long at, uint8_t (&flag)[2]) {  // start the copies of a node row
#pragma unroll
    for (int z = 0; z < 2; ++z) {
      const long long m = at + (z ? sxy : 0);
#pragma unroll
      for (int f = 0; f < 5; ++f) {
        R* dst = reinterpret_cast<R*>(&sh[b].n[f * 2 + z][lane]);
        if (TR::TWO) {
          copy_async(dst, x + f * d.Nn + m);
          copy_async(dst + 1, v + f * d.Nn + m);
        } else {
          copy_async(dst, (TR::DIR ? v : x) + f * d.Nn + m);
        }
        if (TR::VEL && f < 3) copy_async(&sh[b].u[f * 2 + z][lane], x + f * d.Nn + m);
      }
      if (TR::TWO || TR::DIR) flag[z] = d.flag[m];
    }
  };

  const R c0 = R(GW0), c1 = R(GW1);
  Edge<T> lo[5], up[5];
  R s_lo = R(0), s_up = R(0), uv_lo = R(0), uv_up = R(0);  // row sums of u.u and u.v

  auto consume = [&](int b, const uint8_t (&flag)[2], Edge<T> ed[5], R& s2, R& uv) {
    R us = R(0), vs = R(0);
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      T q[2];
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        q[z] = sh[b].n[f * 2 + z][lane];
        const bool masked = (TR::TWO || TR::DIR) && ((flag[z] >> f) & 1);
        if constexpr (TR::TWO)
          q[z].y = masked ? R(0) : q[z].y;  // Dirichlet columns (rows of the adjoint) removed
        else if constexpr (TR::DIR)
          q[z] = masked ? R(0) : q[z];
        if (f < 3) {
          const R u = TR::VEL ? sh[b].u[f * 2 + z][TR::VEL ? lane : 0] : comp<0>(q[z]);
          if (!TR::VEL) us = fma(u, u, us);
          if (K == JVP || K == JVP_LIN) vs = fma(u, TR::TWO ? comp<1>(q[z]) : comp<0>(q[z]), vs);
        }
      }
      ed[f].dz = vsub(q[1], q[0]);
      ed[f].v[0] = vfma(c0, ed[f].dz, q[0]);
      ed[f].v[1] = vfma(c1, ed[f].dz, q[0]);
    }
    s2 = us;
    uv = vs;
  };

  // ---- constants; FP32 weights of a lane without an element are zero
  ElemConst<R> cm = c;
  if (PACKED && !elem) {
    cm.wh = cm.prw = cm.prw2 = cm.wc[0] = cm.wc[1] = R(0);
  }
  Edge<R> carry[5];  // transposed z-stage inputs of the lower node row so far
  R carry_g = R(0);
#pragma unroll
  for (int f = 0; f < 5; ++f) carry[f].dz = carry[f].v[0] = carry[f].v[1] = R(0);
  R* const y0 = TR::TEST ? out + w * (mp.rc + 1) * (long long)ROW_LEN + lane
                         : nullptr;

  issue(0, n, fl0);
  issue(1, n + sx, fl);
  R gam_next = R(0), src_next = R(0);
  auto load_design = [&] {
    if (TR::VEL) return;  // the coefficients come from the store
    gam_next = fresh(gam)[e];
    if (srcs) src_next = fresh(srcs)[e];
  };
  load_design();
  copies_wait();
  consume(0, fl0, lo, s_lo, uv_lo);

  int b = 0;  // buffer of the row below
  auto velocity = [&](int buf, int f, int z) -> R {
    if constexpr (TR::VEL)
      return sh[buf].u[f * 2 + z][lane];
    else
      return comp<0>(sh[buf].n[f * 2 + z][lane]);
  };
  for (int r = 0; r < rows; ++r) {
    const int below = b;
    b = b + 1 == BUFS ? 0 : b + 1;
    copies_wait();
    consume(b, fl, up, s_up, uv_up);
    const R g = gam_next, s = src_next;
    const long long ee = e;
    n += sx;
    e += d.nx;
    if (r + 1 < rows) {
      issue(b + 1 == BUFS ? 0 : b + 1, n + sx, fl);
      load_design();
    }

    // ---- element coefficients
    ElemCoef<R> ks;
    R S = R(0), uv = R(0);
    if constexpr (TR::VEL) {
      ks = lin_coef(cache + ee, d.E, g, s, cm);
    } else {
      S = s_lo + s_up;
      S += shfl(S, to_right);
      ks = coef_of(S, g, s, cm);
    }
    if (K == JVP || K == JVP_LIN) {
      uv = uv_lo + uv_up;
      uv += shfl(uv, to_right);
    }
    R dtau = R(0), dtauT = R(0), da = R(0), dK = R(0);
    if (K == JVP) {  // d tau_e along the direction (scaled units, see elem_jvp)
      dtau = -ks.tau * ks.tau * ks.tau * R(0.0625) * uv;
      dtauT = -ks.tauT * ks.tauT * ks.tauT * R(0.0625) * uv;
    } else if (K == JVP_LIN) {  // the store's ratios dtau/tau (elem_jvp_lin)
      dtau = -ks.tau * ks.tau * R(0.0625) * uv;
      dtauT = -ks.tauT * ks.tauT * R(0.0625) * uv;
    } else if (K == SENS) {  // design derivatives (elem_sens)
      da = c.h * dalpha_of(g, c);
      dK = c.inv_h * dK_of(g, c);
      dtau = -ks.tau * ks.tau * ks.tau * ks.alpha * da;
      dtauT = -ks.tauT * ks.tauT * ks.tauT * ks.K * R(16) * dK;
    }
    R tb = R(0), tbT = R(0), acc = R(0);
    P tb2, tbT2;
    if (PACKED) tb2 = tbT2 = mk(R(0), R(0));

    constexpr int NV = TR::TWO ? 2 : 1;
    P gz[NV][5][2];            // z gradients of the point pairs, by qy (both Gauss planes)
    P BZ[5][2];                // z-gradient fluxes summed over qz
    R vz0[5], vz1[5];          // transposed z-stage inputs of the lower row
#pragma unroll
    for (int qz = 0; qz < 2; ++qz) {
      P val[NV][5][2], gy[NV][5];
      R gx[NV][5][2];
#pragma unroll
      for (int f = 0; f < 5; ++f) {
        const T dy = vsub(up[f].v[qz], lo[f].v[qz]);
        const T a[2] = {vfma(c0, dy, lo[f].v[qz]), vfma(c1, dy, lo[f].v[qz])};
        const T dyn = shfl(dy, to_right), an[2] = {shfl(a[0], to_right), shfl(a[1], to_right)};
        T dz[2], dzn[2];
        if (qz == 0) {
          const T ez = vsub(up[f].dz, lo[f].dz);
          dz[0] = vfma(c0, ez, lo[f].dz);
          dz[1] = vfma(c1, ez, lo[f].dz);
          dzn[0] = shfl(dz[0], to_right);
          dzn[1] = shfl(dz[1], to_right);
        }
        auto stage_x = [&](auto sc) {  // x stage of vector s: values and gradients at the pairs
          constexpr int s_ = decltype(sc)::value;
          {
            const R p = comp<s_>(dy), q = comp<s_>(dyn) - p;
            gy[s_][f] = mk(p + c0 * q, p + c1 * q);
          }
#pragma unroll
          for (int qy = 0; qy < 2; ++qy) {
            const R p = comp<s_>(a[qy]), q = comp<s_>(an[qy]) - p;
            val[s_][f][qy] = mk(p + c0 * q, p + c1 * q);
            gx[s_][f][qy] = q;
            if (qz == 0) {
              const R t = comp<s_>(dz[qy]), u = comp<s_>(dzn[qy]) - t;
              gz[s_][f][qy] = mk(t + c0 * u, t + c1 * u);
            }
          }
        };
        stage_x(std::integral_constant<int, 0>());
        if constexpr (NV == 2) stage_x(std::integral_constant<int, 1>());
      }
      P BY[5];
      R V0[5][2], V1[5][2];  // value slots and x-gradient fluxes on the two faces, by qy
#pragma unroll
      for (int qy = 0; qy < 2; ++qy) {
        const int PI = qy + 2 * qz;
        P f0[5], F1[5][3];
        if constexpr (PACKED) {
          QP2 q, t;
          auto fill = [&](QP2& o, int sv) {
#pragma unroll
            for (int f = 0; f < 3; ++f) {
              o.u[f] = val[sv][f][qy];
              o.G[f][0] = bc2(gx[sv][f][qy]);
              o.G[f][1] = gy[sv][f];
              o.G[f][2] = gz[sv][f][qy];
            }
            o.p = val[sv][3][qy];
            o.gp[0] = bc2(gx[sv][3][qy]);
            o.gp[1] = gy[sv][3];
            o.gp[2] = gz[sv][3][qy];
            o.T = val[sv][4][qy];
            o.gT[0] = bc2(gx[sv][4][qy]);
            o.gT[1] = gy[sv][4];
            o.gT[2] = gz[sv][4][qy];
          };
          fill(q, 0);
          fill(t, 1);
          const Const2 K2 = const2(cm);
          const Coef2 k2 = coef2(ks);
          f2 body[3], rM[3], rT;
          strong_f2(q, k2, K2, body, rM, rT);
          if (TR::ADJ)
            flux_adjoint_f2(q, rM, rT, t, k2, K2, f0, F1, tb2, tbT2);
          else
            flux_tangent_f2(q, rM, rT, t, k2, bc2(cm.wh * dtau), bc2(cm.wh * dtauT), K2, f0, F1);
        } else {
          QP<R> q[2], t[2];
          R rM[2][3], rT[2];
          auto fill = [&](QP<R> o[2], int sv) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              auto at = [&](const P& a) { return h ? a.y : a.x; };
#pragma unroll
              for (int f = 0; f < 3; ++f) {
                o[h].u[f] = at(val[sv][f][qy]);
                o[h].G[f][0] = gx[sv][f][qy];
                o[h].G[f][1] = at(gy[sv][f]);
                o[h].G[f][2] = at(gz[sv][f][qy]);
              }
              o[h].p = at(val[sv][3][qy]);
              o[h].gp[0] = gx[sv][3][qy];
              o[h].gp[1] = at(gy[sv][3]);
              o[h].gp[2] = at(gz[sv][3][qy]);
              o[h].T = at(val[sv][4][qy]);
              o[h].gT[0] = gx[sv][4][qy];
              o[h].gT[1] = at(gy[sv][4]);
              o[h].gT[2] = at(gz[sv][4][qy]);
            }
          };
          if constexpr (TR::DIR) {
            load_lin_pair<R>(cache + ee, d.E, PI, q, rM, rT);
            fill(t, 0);
          } else {
            fill(q, 0);
            if (NV == 2) fill(t, NV - 1);
          }
          R f0s[2][5], F1s[2][5][3];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if constexpr (K == RES) {
              flux_residual(q[h], ks, cm, f0s[h], F1s[h]);
            } else if constexpr (K == JVP) {
              flux_tangent<R, false>(q[h], t[h], ks, R(0), R(0), dtau, dtauT, cm, f0s[h], F1s[h]);
            } else if constexpr (K == JTVP) {
              flux_adjoint(q[h], t[h], ks, cm, f0s[h], F1s[h], tb, tbT);
            } else if constexpr (K == JVP_LIN) {
              flux_tangent_rm<R, false, true>(q[h], rM[h], rT[h], t[h], ks, R(0), R(0), dtau, dtauT,
                                              cm, f0s[h], F1s[h]);
            } else if constexpr (K == JTVP_LIN) {
              flux_adjoint_rm<R, true>(q[h], rM[h], rT[h], t[h], ks, cm, f0s[h], F1s[h], tb, tbT);
            } else if constexpr (K == SENS) {
              acc += point_sens(q[h], t[h], ks, da, dK, dtau, dtauT, cm);
            } else {
              if (elem) store_point(q[h], ks, cm, out + ee + (long long)((2 * PI + h) * LIN_GP) * d.E, d.E);
            }
          }
          if constexpr (TR::TEST) {
#pragma unroll
            for (int f = 0; f < 5; ++f) {
              f0[f] = mk(f0s[0][f], f0s[1][f]);
#pragma unroll
              for (int j = 0; j < 3; ++j) F1[f][j] = mk(F1s[0][f][j], F1s[1][f][j]);
            }
          }
        }
        if constexpr (TR::TEST) {
#pragma unroll
          for (int f = 0; f < 5; ++f) {  // transposed x stage (test8), y and z slots summed
            const R F = F1[f][0].x + F1[f][0].y;
            V1[f][qy] = cm.wc[0] * f0[f].x + (cm.wc[1] * f0[f].y + F);
            V0[f][qy] = cm.wc[1] * f0[f].x + (cm.wc[0] * f0[f].y - F);
            BY[f] = qy ? vadd(BY[f], F1[f][1]) : F1[f][1];
            BZ[f][qy] = qz ? vadd(BZ[f][qy], F1[f][2]) : F1[f][2];
          }
        }
      }
      if constexpr (TR::TEST) {
#pragma unroll
        for (int f = 0; f < 5; ++f) {  // transposed y stage; the faces' two elements added
          const R b1 = c0 * BY[f].x + c1 * BY[f].y, b0 = BY[f].x + BY[f].y - b1;
          R low, high;
          if (PACKED) {
            const P q0 = mk(V0[f][0], V1[f][0]), q1 = mk(V0[f][1], V1[f][1]);
            const P dd = vfma(c1, q1, vfma(c0, q0, mk(b0, b1)));
            const P ll = vsub(vadd(q0, q1), dd);
            low = ll.x + mleft * shfl(ll.y, to_left);
            high = dd.x + mleft * shfl(dd.y, to_left);
          } else {
            auto faces_sum = [&](R a0, R a1) {
              const R t = shfl(a1, to_left);
              return (elem ? a0 : R(0)) + (left ? t : R(0));
            };
            const R q0 = faces_sum(V0[f][0], V1[f][0]), q1 = faces_sum(V0[f][1], V1[f][1]);
            high = faces_sum(b0, b1) + c0 * q0 + c1 * q1;
            low = q0 + q1 - high;
          }
          (qz ? vz1 : vz0)[f] = low + carry[f].v[qz];
          carry[f].v[qz] = high;
        }
      }
    }

    if constexpr (K == SENS) {
      if (elem) out[ee] = acc;
    } else if constexpr (K == LINEARIZE) {
      if (elem) {
        R* o = out + ee + (long long)(8 * LIN_GP) * d.E;
        o[0] = ks.tau;
        o[d.E] = ks.tauT;
        o[2 * d.E] = ks.alpha;
        o[3 * d.E] = ks.K;
      }
    } else {
      R gs = R(0);
      if (TR::ADJ) {  // the tau cotangents reach every velocity row of the element
        if constexpr (PACKED) {
          tb = tb2.x + tb2.y;
          tbT = tbT2.x + tbT2.y;
        }
        R gsum = K == JTVP
            ? -(ks.tau * ks.tau * ks.tau * tb + ks.tauT * ks.tauT * ks.tauT * tbT) * c.wdt
            : -(ks.tau * ks.tau * tb + ks.tauT * ks.tauT * tbT) * R(0.0625);
        const R t = shfl(gsum, to_left);
        gs = (elem ? gsum : R(0)) + (left ? t : R(0));
      }
      R* y = y0 + (long long)r * ROW_LEN;
#pragma unroll
      for (int f = 0; f < 5; ++f) {
        R low, high;
        if (PACKED) {
          P D[2];
#pragma unroll
          for (int qy = 0; qy < 2; ++qy) {
            const R b1 = c0 * BZ[f][qy].x + c1 * BZ[f][qy].y;
            D[qy] = mk(BZ[f][qy].x + BZ[f][qy].y - b1, b1);
          }
          const P ez = vfma(c1, D[1], vfma(c0, D[0], mk(R(0), R(0))));
          const P ll = vsub(vadd(D[0], D[1]), ez);
          low = ll.x + mleft * shfl(ll.y, to_left);
          high = ez.x + mleft * shfl(ez.y, to_left);
        } else {
          R D[2];
#pragma unroll
          for (int qy = 0; qy < 2; ++qy) {
            const R b1 = c0 * BZ[f][qy].x + c1 * BZ[f][qy].y, b0 = BZ[f][qy].x + BZ[f][qy].y - b1;
            const R t = shfl(b1, to_left);
            D[qy] = (elem ? b0 : R(0)) + (left ? t : R(0));
          }
          high = c0 * D[0] + c1 * D[1];
          low = D[0] + D[1] - high;
        }
        const R dzl = low + carry[f].dz;
        carry[f].dz = high;
        R o1 = dzl + c0 * vz0[f] + c1 * vz1[f];
        R o0 = vz0[f] + vz1[f] - o1;
        if (TR::ADJ && f < 3) {
          o0 += (gs + carry_g) * velocity(below, f, 0);
          o1 += (gs + carry_g) * velocity(below, f, 1);
        }
        y[f * 32] = o0;
        y[(5 + f) * 32] = o1;
      }
      carry_g = gs;
    }
#pragma unroll
    for (int f = 0; f < 5; ++f) lo[f] = up[f];
    s_lo = s_up;
    uv_lo = uv_up;
  }
  if constexpr (TR::TEST) {  // the chunk's last node row
    R* y = y0 + (long long)rows * ROW_LEN;
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      R o1 = carry[f].dz + c0 * carry[f].v[0] + c1 * carry[f].v[1];
      R o0 = carry[f].v[0] + carry[f].v[1] - o1;
      if (TR::ADJ && f < 3) {
        o0 += carry_g * velocity(b, f, 0);
        o1 += carry_g * velocity(b, f, 1);
      }
      y[f * 32] = o0;
      y[(5 + f) * 32] = o1;
    }
  }
}

// Sums of node (i, j, k) over its (up to four) faces: the element layers k - 1 and k,
// each one slot, plus the slots of a face shared by two chunks or of a node row shared
// by two runs, in a fixed order.
template <typename R>
__device__ __forceinline__ void node_sums(const LevelDev& d, const MarchPlan& mp, int i, int j, int k,
                                          const R* __restrict__ Y, R acc[5]) {
  const int run = min(j / mp.rc, mp.runs - 1), r = j - run * mp.rc;
  const bool second = r == 0 && run > 0;  // also the last row of the run before
  const int rows = mp.rc + 1;
#pragma unroll
  for (int z = 1; z >= 0; --z) {  // node k is corner z of layer k - z
    const int kz = k - z;
    if (kz < 0 || kz >= d.nz) continue;
    for (int t = 0; t <= (second ? 1 : 0); ++t) {
      const long long l = i + (long long)(d.nx + 1) * (kz + (mp.flat ? d.nz * (long long)(run - t) : 0));
      const long long chunk = l <= 0xffffffffLL ? (unsigned)l / (unsigned)mp.stride : l / mp.stride;
      const int lane = (int)(l - chunk * mp.stride);
      const long long w = chunk + (mp.flat ? 0 : (run - t) * mp.nchunk);
      const R* p = Y + (w * rows + (t ? mp.rc : r)) * ROW_LEN + z * 160 + lane;
#pragma unroll
      for (int f = 0; f < 5; ++f) acc[f] += __ldcg(p + f * 32);  // read once
      if (lane == 0 && i > 0) {  // the left element's share, in lane 31 of the chunk before
        p += mp.stride - (long long)rows * ROW_LEN;
#pragma unroll
        for (int f = 0; f < 5; ++f) acc[f] += __ldcg(p + f * 32);  // read once
      }
    }
  }
}

}  // namespace march
}  // namespace nc
