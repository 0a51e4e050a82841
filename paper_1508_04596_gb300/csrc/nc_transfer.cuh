// Transfers between a fine level and the next coarser one (factor 2), one value.
// 1-D Q1 prolongation weight of coarse node I for fine node i: 1 if i == 2I,
// 1/2 if |i - 2I| == 1.
#pragma once
#include "nc_internal.cuh"

namespace nc {

// Field q of the restriction at coarse node (I, J, K) with flags cfl; rf: the fine
// field.  Fine Dirichlet rows are dropped, coarse ones zero.
template <typename R>
__device__ __forceinline__ R restrict_value(const LevelDev& f, const R* rf, int q, uint8_t cfl, int I, int J,
                                            int K) {
  if ((cfl >> q) & 1) return R(0);
  R acc = R(0);
#pragma unroll
  for (int dk = -1; dk <= 1; ++dk) {
    const int k = 2 * K + dk;
    if (k < 0 || k > f.nz) continue;
#pragma unroll
    for (int dj = -1; dj <= 1; ++dj) {
      const int j = 2 * J + dj;
      if (j < 0 || j > f.ny) continue;
#pragma unroll
      for (int di = -1; di <= 1; ++di) {
        const int i = 2 * I + di;
        if (i < 0 || i > f.nx) continue;
        const R w = R((dk ? 0.5 : 1.0) * (dj ? 0.5 : 1.0) * (di ? 0.5 : 1.0));
        const long long m = i + (long long)(f.nx + 1) * (j + (long long)(f.ny + 1) * k);
        const R v = rf[m];
        if (!((f.flag[m] >> q) & 1)) acc += w * v;
      }
    }
  }
  return acc;
}

// Trilinear prolongation of the coarse field z at fine node (i, j, k).
template <typename R>
__device__ __forceinline__ R prolong_value(const LevelDev& c, const R* z, int i, int j, int k) {
  const int i0 = i >> 1, i1 = (i + 1) >> 1, j0 = j >> 1, j1 = (j + 1) >> 1, k0 = k >> 1, k1 = (k + 1) >> 1;
  R acc = R(0);
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    if (a && k1 == k0) continue;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      if (b && j1 == j0) continue;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        if (e && i1 == i0) continue;
        acc += z[(e ? i1 : i0) + (long long)(c.nx + 1) * ((b ? j1 : j0) + (long long)(c.ny + 1) * (a ? k1 : k0))];
      }
    }
  }
  return acc * R(((i & 1) ? 0.5 : 1.0) * ((j & 1) ? 0.5 : 1.0) * ((k & 1) ? 0.5 : 1.0));
}

}  // namespace nc
