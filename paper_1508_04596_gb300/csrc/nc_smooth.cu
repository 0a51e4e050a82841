// Kernels of the Jacobi-GMRES smoother beyond the vector operations of nc_blas.cu.
#include "nc_smooth.cuh"

namespace nc {

namespace {

// The columns and norms staged in shared memory, then one warp's solve.
__global__ void __launch_bounds__(32) k_small_ls(double* Hd, int k) {
  extern __shared__ double sh[];
  double* H = sh;                   // k columns of k + 1
  double* sig2 = H + k * (k + 1);   // k + 1 each
  double* isig = sig2 + k + 1;
  double* g = isig + k + 1;
  for (int t = threadIdx.x; t < k * (k + 1); t += 32) H[t] = Hd[(t / (k + 1)) * LDH + t % (k + 1)];
  for (int t = threadIdx.x; t <= k; t += 32) {
    sig2[t] = Hd[HD_SIG2 + t];
    isig[t] = Hd[HD_ISIG + t];
  }
  __syncwarp();
  warp_least_squares(k, H, k + 1, sig2, isig, Hd + HD_Y, g);
}

}  // namespace

void small_ls(double* Hd, int k, cudaStream_t s) {
  // at most (64 + 3) * 65 doubles, below the 48 KB a kernel has without asking
  k_small_ls<<<1, 32, sizeof(double) * (k + 3) * (k + 1), s>>>(Hd, k);
}

}  // namespace nc
