// Rows of the element Jacobians from the linearisation store, added into the stencil.
//
// A launch takes one local test node a and a thread per element: the rows (f, a),
// f = 0..4, of J_e against all 40 unknowns (g, b).  With the point quantities of the
// store (u, G = h grad u, h grad T, the SUPG weights rM = wtau rM, rT = wtauT rT), the
// test values N_a, D_a = h grad N_a at the points, U_a = u . D_a, W = wh N_a + wtau U_a
// and W' = wh N_a + wtauT U_a, the entries are (sums over the points; from
// flux_tangent_rm with the direction N_b, D_b)
//   (i, g):  (W G_ig + D_ag rM_i) N_b + delta_ig W (u . D_b + alpha N_b)
//              + prw (delta_ig D_a . D_b + D_ag D_bi) - tau^2/16 (U_a rM_i) u_bg
//   (i, p):  wtau U_a D_bi - wh D_ai N_b          (i, T):  beg_i W N_b
//   (p, g):  wtau [(D_a . G_g + alpha D_ag) N_b + D_ag u . D_b] + wh N_a D_bg
//              - tau^2/16 (D_a . rM) u_bg
//   (p, p):  wtau D_a . D_b                        (p, T):  wtau (beg . D_a) N_b
//   (T, g):  (W' gT_g + D_ag rT) N_b - tauT^2/16 (U_a rT) u_bg
//   (T, T):  W' u . D_b + wK D_a . D_b             (T, p):  0
// The sums over the 8 points against N_b for the 8 nodes b are tensor products: with
// 1-D weights s (same side) and c (other side) factored as s (1, c/s), a stage is two
// FMAs per pair, 24 for all b (64 one by one); against D_bk 12, since D_bk is a sign
// along axis k.  Products of test and trial functions alone (the viscous, pressure
// and mass terms) are constants.  About 1,500 FP64 operations per element and test
// node, 12,000 per element, where 40 products with unit directions took 32,000 (64^3:
// 15.4 ms FP64, with their rows written, read and added; now 6.9.  FP32 2.7 -> 1.5).
//
// Every entry of the stencil gets at most one contribution from a launch (the
// element and a fix its node, b its offset), so the reductions to memory (no return,
// the addition happens in L2 and off the FP64 pipe) leave a result that depends on
// the order of the eight launches alone.
#pragma once
#include "nc_internal.cuh"

namespace nc {
namespace rows {

constexpr double RHO = GW0 / GW1;  // c / s

// v[b] <- sum_p v[p] prod rho(b, p), rho = 1 on the same side of an axis, c/s on the other
template <typename R>
__device__ __forceinline__ void against_N(R v[8]) {
  const R r = R(RHO);
#pragma unroll
  for (int st = 1; st < 8; st *= 2)
#pragma unroll
    for (int p = 0; p < 8; ++p)
      if (!(p & st)) {
        const R a = v[p], b = v[p + st];
        v[p] = fma(r, b, a);
        v[p + st] = fma(r, a, b);
      }
}

// w[j] <- the same without axis K (whose points are summed), j = the two other bits of
// b in ascending axis order; the entry of node b is w times the sign of b along K
template <typename R, int K>
__device__ __forceinline__ void against_D(const R v[8], R w[4]) {
  const R r = R(RHO);
  constexpr int st = 1 << K, s0 = K == 0 ? 2 : 1, s1 = K == 2 ? 2 : 4;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int p = (j & 1 ? s0 : 0) + (j & 2 ? s1 : 0);
    w[j] = v[p] + v[p + st];
  }
#pragma unroll
  for (int t = 1; t < 4; t *= 2)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (!(j & t)) {
        const R a = w[j], b = w[j + t];
        w[j] = fma(r, b, a);
        w[j + t] = fma(r, a, b);
      }
}
// index into against_D's result and sign of node b
template <int K> __device__ __forceinline__ constexpr int dj(int b) {
  return K == 0 ? b >> 1 : (K == 1 ? (b & 1) + ((b >> 2) << 1) : b & 3);
}
template <typename R, int K> __device__ __forceinline__ R dsign(int b, R v) { return (b >> K) & 1 ? v : -v; }

// Sums over the points of products of test and trial functions alone, for test node a
// and every trial node b (kernel arguments: operands that cost no instruction):
// vv = prw (D_a . D_b delta_ig + D_ag D_bi), dn = D_ag N_b, pv = wh N_a D_bg,
// vp = -wh D_ai N_b, pT = (beg . D_a) N_b, lap = D_a . D_b.
template <typename R>
struct RowConst {
  R vv[3][3][8], dn[3][8], pv[3][8], vp[3][8], pT[8], lap[8];
};

template <typename R>
RowConst<R> row_const(const ElemConst<R>& c, int a) {
  RowConst<R> k;
  auto bit = [](int n, int t) { return (n >> t) & 1; };
  auto sg = [&](int n, int t) { return bit(n, t) ? 1.0 : -1.0; };
  auto mass = [&](int t, int b) { return bit(a, t) == bit(b, t) ? 2.0 / 3.0 : 1.0 / 3.0; };
  for (int b = 0; b < 8; ++b) {
    double lap = 0.0, pT = 0.0;
    for (int g = 0; g < 3; ++g) {
      const int t0 = g == 0 ? 1 : 0, t1 = g == 2 ? 1 : 2;
      const double mm = mass(t0, b) * mass(t1, b);
      lap += 2.0 * sg(a, g) * sg(b, g) * mm;
      k.dn[g][b] = R(sg(a, g) * mm);
      k.pv[g][b] = R((double)c.wh * sg(b, g) * mm);
      k.vp[g][b] = R(-(double)c.wh * sg(a, g) * mm);
      pT += (double)c.beg[g] * sg(a, g) * mm;
    }
    k.lap[b] = R(lap);
    k.pT[b] = R(pT);
    for (int i = 0; i < 3; ++i)
      for (int g = 0; g < 3; ++g) {
        const int t0 = g == 0 ? 1 : 0, t1 = g == 2 ? 1 : 2;
        const double dd = i == g ? 2.0 * sg(a, g) * sg(b, g) * mass(t0, b) * mass(t1, b) + lap
                                 : sg(a, g) * sg(b, i) * mass(3 - g - i, b);
        k.vv[i][g][b] = R((double)c.prw * dd);
      }
  }
  return k;
}

// FP64 keeps 168 registers (three blocks), FP32 takes 255 (two).  The whole assembly at 64^3 in
// FP64: 6.89 ms, 6.82 with two blocks; in FP32: 1.49 ms, 1.41 with three, 2.20 with four.
template <typename R>
__global__ void __launch_bounds__(128, sizeof(R) == 8 ? 3 : 2)
    k_assemble_rows(LevelDev d, ElemConst<R> c, RowConst<R> kc, const R* __restrict__ x,
                    const R* __restrict__ cache, int a, R* S) {
  const long long e = blockIdx.x * 128LL + threadIdx.x;
  if (e >= d.E) return;
  int ei, ej, ek;
  elem_ijk(d, e, ei, ej, ek);
  const long long sy = d.nx + 1, sz = (long long)(d.nx + 1) * (d.ny + 1);
  const long long n0 = ei + sy * (ej + (long long)(d.ny + 1) * ek);
  const int ab[3] = {a & 1, (a >> 1) & 1, a >> 2};
  const long long na = n0 + ab[0] + ab[1] * sy + ab[2] * sz;
  const unsigned row_flag = d.flag[na];
  unsigned col_flag[8];
#pragma unroll
  for (int b = 0; b < 8; ++b) col_flag[b] = d.flag[n0 + (b & 1) + ((b >> 1) & 1) * sy + (b >> 2) * sz];

  const long long E = d.E;
  const R* const st = cache + e;
  auto lin = [&](int p, int q) { return st[(long long)(p * LIN_GP + q) * E]; };
  const R tau = st[(long long)(8 * LIN_GP) * E], tauT = st[(long long)(8 * LIN_GP + 1) * E];
  const R alpha = st[(long long)(8 * LIN_GP + 2) * E], Kc = st[(long long)(8 * LIN_GP + 3) * E];
  const R wtau = c.wh * tau, wtauT = c.wh * tauT, wK = c.wh * Kc;

  // ---- test function: 1-D values and signed products
  R w1[3][2], E1[3][4];  // n(a, q) per axis; D_a along axis g on the other axes' points
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    w1[t][0] = ab[t] ? R(GW0) : R(GW1);
    w1[t][1] = ab[t] ? R(GW1) : R(GW0);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int lo = j & 1, hi = j >> 1;
    E1[0][j] = (ab[0] ? w1[1][lo] : -w1[1][lo]) * w1[2][hi];
    E1[1][j] = (ab[1] ? w1[0][lo] : -w1[0][lo]) * w1[2][hi];
    E1[2][j] = (ab[2] ? w1[0][lo] : -w1[0][lo]) * w1[1][hi];
  }
  auto D = [&](int g, int p) { return E1[g][g == 0 ? p >> 1 : (g == 1 ? (p & 1) + ((p >> 2) << 1) : p & 3)]; };

  // s^3 and s^2 of the factored weights go into the last operation on a sum
  const R S3 = R(GW1 * GW1 * GW1), S2 = R(GW1 * GW1);
  R U[8], W[8], WT[8];
  R tp = R(0), tT = R(0), tm[3] = {R(0), R(0), R(0)};
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const R Na = E1[2][p & 3] * (ab[2] ? w1[2][p >> 2] : -w1[2][p >> 2]);
    U[p] = lin(p, 0) * D(0, p) + lin(p, 1) * D(1, p) + lin(p, 2) * D(2, p);
    const R wn = c.wh * Na;
    W[p] = fma(wtau, U[p], wn);
    WT[p] = fma(wtauT, U[p], wn);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const R rm = lin(p, 15 + i);
      tm[i] = fma(U[p], rm, tm[i]);
      tp = fma(D(i, p), rm, tp);
    }
    tT = fma(U[p], lin(p, 18), tT);
  }
  const R q2 = -(tau * tau) * R(0.0625), q2T = -(tauT * tauT) * R(0.0625);
  tp *= q2;
  tT *= q2T;
#pragma unroll
  for (int i = 0; i < 3; ++i) tm[i] *= q2;

  auto add = [&](int f, int g, int b, R v) {
    if (((row_flag >> f) & 1) || ((col_flag[b] >> g) & 1)) return;
    const int o = ((b & 1) - ab[0] + 1) + 3 * (((b >> 1) & 1) - ab[1] + 1) + 9 * ((b >> 2) - ab[2] + 1);
    atomicAdd(S + ((long long)(o * 5 + f) * 5 + g) * d.Nn + na, v);
  };
  auto xb = [&](int g, int b) { return x[g * d.Nn + n0 + (b & 1) + ((b >> 1) & 1) * sy + (b >> 2) * sz]; };

  // sum of w u . D_b for the point weights w, over s^2
  auto convect = [&](auto w, R out[8]) {
    R v[8], y[4];
#pragma unroll
    for (int p = 0; p < 8; ++p) v[p] = w(p) * lin(p, 0);
    against_D<R, 0>(v, y);
#pragma unroll
    for (int b = 0; b < 8; ++b) out[b] = dsign<R, 0>(b, y[dj<0>(b)]);
#pragma unroll
    for (int p = 0; p < 8; ++p) v[p] = w(p) * lin(p, 1);
    against_D<R, 1>(v, y);
#pragma unroll
    for (int b = 0; b < 8; ++b) out[b] += dsign<R, 1>(b, y[dj<1>(b)]);
#pragma unroll
    for (int p = 0; p < 8; ++p) v[p] = w(p) * lin(p, 2);
    against_D<R, 2>(v, y);
#pragma unroll
    for (int b = 0; b < 8; ++b) out[b] += dsign<R, 2>(b, y[dj<2>(b)]);
  };

  // ---- temperature columns and the convection of the momentum diagonal
  R C[8];  // over s^3
  convect([&](int p) { return W[p]; }, C);
  {
    R X[8];
#pragma unroll
    for (int p = 0; p < 8; ++p) X[p] = W[p];
    against_N(X);
#pragma unroll
    for (int b = 0; b < 8; ++b) C[b] = fma(alpha, X[b], C[b] * R(1.0 / GW1));
#pragma unroll
    for (int i = 0; i < 3; ++i)
      if (c.beg[i] != R(0)) {
        const R k = S3 * c.beg[i];
#pragma unroll
        for (int b = 0; b < 8; ++b) add(i, 4, b, k * X[b]);
      }
  }
  // ---- momentum rows, velocity columns
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int g = 0; g < 3; ++g) {
      R v[8];
#pragma unroll
      for (int p = 0; p < 8; ++p) v[p] = fma(W[p], lin(p, 3 + 3 * i + g), D(g, p) * lin(p, 15 + i));
      against_N(v);
#pragma unroll
      for (int b = 0; b < 8; ++b)
        add(i, g, b, fma(S3, i == g ? v[b] + C[b] : v[b], fma(tm[i], xb(g, b), kc.vv[i][g][b])));
    }
  // ---- momentum rows, pressure columns
  {
    const R k = wtau * S2;
    R y[4];
    against_D<R, 0>(U, y);
#pragma unroll
    for (int b = 0; b < 8; ++b) add(0, 3, b, fma(dsign<R, 0>(b, y[dj<0>(b)]), k, kc.vp[0][b]));
    against_D<R, 1>(U, y);
#pragma unroll
    for (int b = 0; b < 8; ++b) add(1, 3, b, fma(dsign<R, 1>(b, y[dj<1>(b)]), k, kc.vp[1][b]));
    against_D<R, 2>(U, y);
#pragma unroll
    for (int b = 0; b < 8; ++b) add(2, 3, b, fma(dsign<R, 2>(b, y[dj<2>(b)]), k, kc.vp[2][b]));
  }
  // ---- continuity row
  {
    const R k3 = wtau * S3, k2 = wtau * S2, ka = wtau * alpha;
#pragma unroll
    for (int g = 0; g < 3; ++g) {
      R v[8], o[8];
#pragma unroll
      for (int p = 0; p < 8; ++p)
        v[p] = D(0, p) * lin(p, 3 + g) + D(1, p) * lin(p, 6 + g) + D(2, p) * lin(p, 9 + g);
      against_N(v);
      convect([&](int p) { return D(g, p); }, o);
#pragma unroll
      for (int b = 0; b < 8; ++b)
        add(3, g, b, fma(k3, v[b], fma(k2, o[b], fma(ka, kc.dn[g][b], fma(tp, xb(g, b), kc.pv[g][b])))));
    }
  }
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    add(3, 3, b, wtau * kc.lap[b]);
    add(3, 4, b, wtau * kc.pT[b]);
  }
  // ---- energy row
#pragma unroll
  for (int g = 0; g < 3; ++g) {
    R v[8];
#pragma unroll
    for (int p = 0; p < 8; ++p) v[p] = fma(WT[p], lin(p, 12 + g), D(g, p) * lin(p, 18));
    against_N(v);
#pragma unroll
    for (int b = 0; b < 8; ++b) add(4, g, b, fma(S3, v[b], tT * xb(g, b)));
  }
  {
    R o[8];
    convect([&](int p) { return WT[p]; }, o);
#pragma unroll
    for (int b = 0; b < 8; ++b) add(4, 4, b, fma(S2, o[b], wK * kc.lap[b]));
  }
}

}  // namespace rows
}  // namespace nc
