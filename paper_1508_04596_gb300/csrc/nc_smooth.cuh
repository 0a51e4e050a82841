// The small least-squares problem of the Jacobi-GMRES smoother, by one warp.
#pragma once
#include "nc_internal.cuh"

namespace nc {

// Column j of H (leading dimension ld, in shared memory) holds the raw dots
// g_ij = <v_i, w_j> (i <= j) of the unnormalised basis v_i with squared norms
// sig2_i, built so that  A D^-1 v_j = sum_i g_ij / sig2_i v_i + sigma_j v_{j+1}.  With
// q_i = v_i / sigma_i this is the usual Arnoldi relation with the Hessenberg entries
// g_ij / (sigma_i sigma_j) and sigma_{j+1} below the diagonal, and beta = sigma_0.
// Solves min || beta e1 - H y || by Givens rotations in place and leaves y_j / sigma_j,
// the coefficients of the correction on the raw basis, in y.  A vanishing norm or
// pivot (an exhausted Krylov space) contributes zero.
//
// Called by the 32 lanes of one warp; a rotation is formed by all lanes and applied
// by lane j to column j (and j + 32), the substitution runs by columns with a lane per
// row.  An FP64 instruction takes a scheduler 64 cycles whatever the number of active
// lanes: one thread working through the k^2 operations took 40 us for k = 6, this
// 6 us.  isig: the norms' reciprocal roots, 0 where they vanish; g (k + 1) is scratch.
__device__ __forceinline__ void warp_least_squares(int k, double* H, int ld, const double* sig2,
                                                   const double* isig, double* y, double* g) {
  const int lane = threadIdx.x & 31;
  for (int i = lane; i <= k; i += 32) g[i] = 0.0;
  __syncwarp();
  if (lane == 0) {
    const double b2 = sig2[0], beta = sqrt(b2 > 0.0 ? b2 : 0.0);
    g[0] = (beta > 0.0 && beta < 1e300) ? beta : 0.0;
  }
  for (int j = lane; j < k; j += 32) {  // raw dots -> normalised Hessenberg
    double* h = H + (long long)j * ld;
    const double ij = isig[j];
    for (int i = 0; i <= j; ++i) h[i] *= isig[i] * ij;
    const double s2 = sig2[j + 1];
    h[j + 1] = ij > 0.0 ? sqrt(s2 > 0.0 ? s2 : 0.0) : 0.0;
  }
  __syncwarp();
  double rmax = 0.0;
  for (int q = 0; q < k; ++q) {
    const double a = H[q * ld + q], b = H[q * ld + q + 1];
    const double r2 = a * a + b * b;
    double r, ir;
    if (r2 > 1e-280 && r2 < 1e280) {
      ir = rsqrt(r2);
      r = r2 * ir;
    } else {  // out of the range of the squares (or exhausted, or not finite)
      r = hypot(a, b);
      ir = r > 0.0 ? 1.0 / r : 0.0;
    }
    const double c = r > 0.0 ? a * ir : 1.0, s = r > 0.0 ? b * ir : 0.0;
    rmax = fmax(rmax, r);
    __syncwarp();
    for (int j = q + 1 + lane; j <= k; j += 32) {  // column k stands for the right-hand side
      double* h = j < k ? H + j * ld : g;
      const double t1 = h[q], t2 = h[q + 1];
      h[q] = c * t1 + s * t2;
      h[q + 1] = c * t2 - s * t1;
    }
    if (lane == 0) {
      H[q * ld + q] = r;
      H[q * ld + q + 1] = ir;  // kept for the substitution
    }
    __syncwarp();
  }
  for (int j = k - 1; j >= 0; --j) {
    const double acc = g[j], r = H[j * ld + j];
    const double v = (r > 1e-14 * rmax && isfinite(acc)) ? acc * H[j * ld + j + 1] : 0.0;
    __syncwarp();
    if (lane == 0) y[j] = v * isig[j];
    for (int i = lane; i < j; i += 32) g[i] -= H[j * ld + i] * v;
    __syncwarp();
  }
}

}  // namespace nc
