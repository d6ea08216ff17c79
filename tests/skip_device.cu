// Device build of the z pass's skip test (csrc/collapse_x2.cuh) and of the
// collapse time that it may not lose: FP32 in packed pairs, from the FP32
// eigenvalues in FP64 where the root is ill-conditioned, as the kernels do it.
#include <cuda_runtime.h>

#include "collapse.cuh"
#include "collapse_x2.cuh"

__global__ void k_skip(const float* lam, const float* fm, int n, int nf, int corr, double dcorr, float tau,
                       unsigned char* cleared, float* F) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n / 2) return;
  const int j[2] = {i, i + n / 2};
  float2 l[3];
  for (int k = 0; k < 3; ++k) l[k] = make_float2(lam[3 * j[0] + k], lam[3 * j[1] + k]);
  const pin::CollapseConsts<float> cc{(float)dcorr, corr};
  const pin::CollapseConsts<double> ccd{dcorr, corr};
  float2 kap;
  const float2 f = pin::collapse_from_eigs_x2(l, cc, kap);
  for (int u = 0; u < 2; ++u) {
    F[j[u]] = u ? f.y : f.x;
    if ((u ? kap.y : kap.x) < tau) {
      const double d[3] = {lam[3 * j[u]], lam[3 * j[u] + 1], lam[3 * j[u] + 2]};
      double k64;
      F[j[u]] = (float)pin::collapse_from_eigs<double>(d, ccd, k64);
    }
  }
  for (int q = 0; q < nf; ++q) {
    const unsigned c = pin::cannot_beat_x2<true>(l, cc, make_float2(fm[(size_t)q * n + j[0]], fm[(size_t)q * n + j[1]]));
    cleared[(size_t)q * n + j[0]] = c & 1u;
    cleared[(size_t)q * n + j[1]] = (c >> 1) & 1u;
  }
}

// n even; fm and cleared are [nf][n]
extern "C" int dev_skip(const float* lam, const float* fm, int n, int nf, int corr, double dcorr, float tau,
                        unsigned char* cleared, float* F) {
  float *dl, *dm, *dF;
  unsigned char* dc;
  const size_t m = (size_t)n * nf;
  if (cudaMalloc(&dl, 12 * (size_t)n) || cudaMalloc(&dm, 4 * m) || cudaMalloc(&dF, 4 * (size_t)n) || cudaMalloc(&dc, m))
    return 1;
  cudaMemcpy(dl, lam, 12 * (size_t)n, cudaMemcpyHostToDevice);
  cudaMemcpy(dm, fm, 4 * m, cudaMemcpyHostToDevice);
  k_skip<<<(n / 2 + 127) / 128, 128>>>(dl, dm, n, nf, corr, dcorr, tau, dc, dF);
  const int rc = cudaDeviceSynchronize() != cudaSuccess;
  cudaMemcpy(cleared, dc, m, cudaMemcpyDeviceToHost);
  cudaMemcpy(F, dF, 4 * (size_t)n, cudaMemcpyDeviceToHost);
  cudaFree(dl); cudaFree(dm); cudaFree(dF); cudaFree(dc);
  return rc;
}
