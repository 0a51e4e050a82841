// Element operators on small grids: four warps per chunk of faces.
//
// A grid with fewer chunks than the GPU has schedulers leaves most of them idle while
// each busy one works through whole elements (FP64: about 1,150 instructions of 64
// cycles, 38 us for the residual, however small the grid).  Here a quad of warps
// takes one chunk of a flat MarchPlan (one element row), each warp one pair of
// Gauss points (qy, qz) of every element: the stages before the fluxes shrink to what
// the pair needs, and since everything after the fluxes is linear, each warp carries
// its pair's share through to the 20 node sums of its lane; the quad adds them in
// shared memory in warp order.  About 0.35 of the FP64 instructions per warp (residual
// at 12^3 with its gather 27 us, 51 with whole elements), but more in all: on larger
// grids the marching kernels are faster (96^3, FP32 J v: 139 us against 84).
#pragma once
#include "nc_march.cuh"

namespace nc {
namespace march {

template <typename R> struct QuadSums {
  R o[4][20][32];
};

template <typename R, int K>
__global__ void __launch_bounds__(128) k_split(LevelDev d, ElemConst<R> c, MarchPlan mp,
                                               const R* __restrict__ x_, const R* __restrict__ gam,
                                               const R* __restrict__ srcs, const R* __restrict__ cache_,
                                               const R* __restrict__ v_, R* Y) {
  chained();
  const R* const x = fresh(x_);
  const R* const cache = fresh(cache_);
  const R* const v = fresh(v_);
  __shared__ QuadSums<R> sums;
  const long long w = blockIdx.x;  // the chunk
  const int q = threadIdx.x >> 5;  // the warp of the quad
  typedef Traits<K> TR;
  typedef typename Stage<R, K>::T T;
  typedef PR<R> P;
  constexpr bool PACKED = std::is_same<R, float>::value && TR::TWO;
  const int lane = threadIdx.x & 31, qy = q & 1, qz = q >> 1;
  const long long faces = (long long)(d.nx + 1) * d.nz * d.ny;
  const long long l = min(w * mp.stride + lane, faces - 1);
  const bool valid = w * mp.stride + lane < faces;
  int i, k, j;
  split3(l, faces, d.nx + 1, d.nz, i, k, j);
  const bool elem = valid && lane < 31 && i < d.nx;
  const bool left = valid && lane > 0 && i > 0;
  const int to_right = elem ? lane + 1 : lane, to_left = left ? lane - 1 : lane;
  const long long sx = d.nx + 1, sxy = sx * (d.ny + 1);
  const long long n = i + sx * (j + (long long)(d.ny + 1) * k);
  const long long e = min(i, d.nx - 1) + (long long)d.nx * (j + (long long)d.ny * k);
  const R c0 = R(GW0), c1 = R(GW1), cy = qy ? c1 : c0, cz = qz ? c1 : c0;

  // ---- nodal values, z stage (this warp's plane), row sums of u.u and u.v
  T dzr[5][2], vr[5][2];  // [field][row]
  R vel[TR::ADJ ? 3 : 1][2][2];
  R S = R(0), uv = R(0);
  const R g = TR::VEL ? R(0) : fresh(gam)[e], s = TR::VEL || !srcs ? R(0) : fresh(srcs)[e];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    uint8_t fl[2] = {0, 0};
    if (TR::TWO || TR::DIR) {
      fl[0] = d.flag[n + r * sx];
      fl[1] = d.flag[n + r * sx + sxy];
    }
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      T nod[2];
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        const long long at = f * d.Nn + n + r * sx + (z ? sxy : 0);
        const bool masked = (TR::TWO || TR::DIR) && ((fl[z] >> f) & 1);
        R u = R(0), t = R(0);
        if (!TR::DIR || f < 3) u = x[at];
        if (TR::TWO || TR::DIR) {
          t = v[at];
          t = masked ? R(0) : t;
        }
        if constexpr (TR::TWO) nod[z] = mk(u, t);
        else if constexpr (TR::DIR) nod[z] = t;
        else nod[z] = u;
        if (f < 3) {
          if (!TR::VEL) S = fma(u, u, S);
          if (K == JVP || K == JVP_LIN) uv = fma(u, t, uv);
          if (TR::ADJ) vel[TR::ADJ ? f : 0][r][z] = u;
        }
      }
      dzr[f][r] = vsub(nod[1], nod[0]);
      vr[f][r] = vfma(cz, dzr[f][r], nod[0]);
    }
  }

  // ---- element coefficients (as k_march)
  ElemCoef<R> ks;
  if constexpr (TR::VEL) {
    ks = lin_coef(cache + e, d.E, g, s, c);
  } else {
    S += shfl(S, to_right);
    ks = coef_of(S, g, s, c);
  }
  R dtau = R(0), dtauT = R(0);
  if (K == JVP || K == JVP_LIN) {
    uv += shfl(uv, to_right);
    dtau = -(K == JVP ? ks.tau : R(1)) * ks.tau * ks.tau * R(0.0625) * uv;
    dtauT = -(K == JVP ? ks.tauT : R(1)) * ks.tauT * ks.tauT * R(0.0625) * uv;
  }

  // ---- y and x stages of this warp's point pair
  constexpr int NV = TR::TWO ? 2 : 1;
  P val[NV][5], gy[NV][5], gz[NV][5];
  R gx[NV][5];
#pragma unroll
  for (int f = 0; f < 5; ++f) {
    const T dy = vsub(vr[f][1], vr[f][0]), a = vfma(cy, dy, vr[f][0]);
    const T dz = vfma(cy, vsub(dzr[f][1], dzr[f][0]), dzr[f][0]);
    const T dyn = shfl(dy, to_right), an = shfl(a, to_right), dzn = shfl(dz, to_right);
    auto stage_x = [&](auto sc) {
      constexpr int s_ = decltype(sc)::value;
      const R p = comp<s_>(dy), pq = comp<s_>(dyn) - p;
      gy[s_][f] = mk(p + c0 * pq, p + c1 * pq);
      const R u = comp<s_>(a), uq = comp<s_>(an) - u;
      val[s_][f] = mk(u + c0 * uq, u + c1 * uq);
      gx[s_][f] = uq;
      const R t = comp<s_>(dz), tq = comp<s_>(dzn) - t;
      gz[s_][f] = mk(t + c0 * tq, t + c1 * tq);
    };
    stage_x(std::integral_constant<int, 0>());
    if constexpr (NV == 2) stage_x(std::integral_constant<int, 1>());
  }

  // ---- fluxes
  P f0[5], F1[5][3];
  R tb = R(0), tbT = R(0);
  if constexpr (PACKED) {
    QP2 a, t;
    auto fill = [&](QP2& o, int sv) {
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        o.u[f] = val[sv][f];
        o.G[f][0] = bc2(gx[sv][f]);
        o.G[f][1] = gy[sv][f];
        o.G[f][2] = gz[sv][f];
      }
      o.p = val[sv][3];
      o.gp[0] = bc2(gx[sv][3]);
      o.gp[1] = gy[sv][3];
      o.gp[2] = gz[sv][3];
      o.T = val[sv][4];
      o.gT[0] = bc2(gx[sv][4]);
      o.gT[1] = gy[sv][4];
      o.gT[2] = gz[sv][4];
    };
    fill(a, 0);
    fill(t, 1);
    const Const2 K2 = const2(c);
    const Coef2 k2 = coef2(ks);
    f2 body[3], rM[3], rT;
    strong_f2(a, k2, K2, body, rM, rT);
    if (TR::ADJ) {
      f2 b2 = mk(0.0f, 0.0f), bT2 = b2;
      flux_adjoint_f2(a, rM, rT, t, k2, K2, f0, F1, b2, bT2);
      tb = b2.x + b2.y;
      tbT = bT2.x + bT2.y;
    } else {
      flux_tangent_f2(a, rM, rT, t, k2, bc2(c.wh * dtau), bc2(c.wh * dtauT), K2, f0, F1);
    }
  } else {
    QP<R> a[2], t[2];
    R rM[2][3], rT[2];
    auto fill = [&](QP<R> o[2], int sv) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        auto at = [&](const P& b) { return h ? b.y : b.x; };
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          o[h].u[f] = at(val[sv][f]);
          o[h].G[f][0] = gx[sv][f];
          o[h].G[f][1] = at(gy[sv][f]);
          o[h].G[f][2] = at(gz[sv][f]);
        }
        o[h].p = at(val[sv][3]);
        o[h].gp[0] = gx[sv][3];
        o[h].gp[1] = at(gy[sv][3]);
        o[h].gp[2] = at(gz[sv][3]);
        o[h].T = at(val[sv][4]);
        o[h].gT[0] = gx[sv][4];
        o[h].gT[1] = at(gy[sv][4]);
        o[h].gT[2] = at(gz[sv][4]);
      }
    };
    if constexpr (TR::DIR) {
      load_lin_pair<R>(cache + e, d.E, q, a, rM, rT);
      fill(t, 0);
    } else {
      fill(a, 0);
      if (NV == 2) fill(t, NV - 1);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      R f0s[5], F1s[5][3];
      if constexpr (K == RES)
        flux_residual(a[h], ks, c, f0s, F1s);
      else if constexpr (K == JVP)
        flux_tangent<R, false>(a[h], t[h], ks, R(0), R(0), dtau, dtauT, c, f0s, F1s);
      else if constexpr (K == JTVP)
        flux_adjoint(a[h], t[h], ks, c, f0s, F1s, tb, tbT);
      else if constexpr (K == JVP_LIN)
        flux_tangent_rm<R, false, true>(a[h], rM[h], rT[h], t[h], ks, R(0), R(0), dtau, dtauT, c, f0s, F1s);
      else
        flux_adjoint_rm<R, true>(a[h], rM[h], rT[h], t[h], ks, c, f0s, F1s, tb, tbT);
#pragma unroll
      for (int f = 0; f < 5; ++f) {
        (h ? f0[f].y : f0[f].x) = f0s[f];
#pragma unroll
        for (int jj = 0; jj < 3; ++jj) (h ? F1[f][jj].y : F1[f][jj].x) = F1s[f][jj];
      }
    }
  }

  // ---- transposed stages of the pair, through to the node sums
  auto faces_sum = [&](R a0, R a1) {
    const R t = shfl(a1, to_left);
    return (elem ? a0 : R(0)) + (left ? t : R(0));
  };
  R gs = R(0);
  if (TR::ADJ) {
    const R gsum = K == JTVP
        ? -(ks.tau * ks.tau * ks.tau * tb + ks.tauT * ks.tauT * ks.tauT * tbT) * c.wdt
        : -(ks.tau * ks.tau * tb + ks.tauT * ks.tauT * tbT) * R(0.0625);
    gs = faces_sum(gsum, gsum);
  }
#pragma unroll
  for (int f = 0; f < 5; ++f) {
    const R F = F1[f][0].x + F1[f][0].y;
    const R V = faces_sum(c.wc[1] * f0[f].x + (c.wc[0] * f0[f].y - F), c.wc[0] * f0[f].x + (c.wc[1] * f0[f].y + F));
    const R by = c0 * F1[f][1].x + c1 * F1[f][1].y, bz = c0 * F1[f][2].x + c1 * F1[f][2].y;
    const R B = faces_sum(F1[f][1].x + F1[f][1].y - by, by), Z = faces_sum(F1[f][2].x + F1[f][2].y - bz, bz);
    const R high = B + cy * V, low = V - high;
    const R zu = cy * Z, zl = Z - zu;
    R o[2][2];  // [row][z]
    o[1][1] = zu + cz * high;
    o[1][0] = high - o[1][1];
    o[0][1] = zl + cz * low;
    o[0][0] = low - o[0][1];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        if (TR::ADJ && f < 3) o[r][z] += gs * vel[f < 3 && TR::ADJ ? f : 0][r][z];
        sums.o[q][(r * 2 + z) * 5 + f][lane] = o[r][z];
      }
  }
  __syncthreads();
  // warp q adds the five sums of node row q / 2, corner q % 2
  R* y = Y + w * 2 * (long long)ROW_LEN + (q >> 1) * ROW_LEN + (q & 1) * 160 + lane;
#pragma unroll
  for (int f = 0; f < 5; ++f)
    y[f * 32] = (sums.o[0][q * 5 + f][lane] + sums.o[1][q * 5 + f][lane]) +
                (sums.o[2][q * 5 + f][lane] + sums.o[3][q * 5 + f][lane]);
}

}  // namespace march
}  // namespace nc
