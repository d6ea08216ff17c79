// The particle order of csrc/fragment.cu behind a host function, so that tests
// can give it any F_max: every number of passes and width of digits.
#include "fragment.cu"

// Returns the passes that the sort took, or -1.  nz a multiple of 4.
extern "C" int dev_order(const float* F, int nx, int ny, int nz, int* order, unsigned char* n_before, int* width) {
  const long n = (long)nx * ny * nz;
  float* dF = nullptr;
  int *dorder = nullptr, *derr = nullptr;
  unsigned char* dn = nullptr;
  char* scratch = nullptr;
  if (cudaMalloc(&dF, n * 4) || cudaMalloc(&dorder, n * 4) || cudaMalloc(&derr, 4) || cudaMalloc(&dn, n) ||
      cudaMalloc(&scratch, pin::fragment_scratch_bytes(n)))
    return -1;
  cudaMemcpy(dF, F, n * 4, cudaMemcpyHostToDevice);
  cudaMemset(derr, 0, 4);
  int rc = pin::fragment_order(dF, nx, ny, nz, scratch, dorder, dn, 0, derr, nullptr) != cudaSuccess;
  rc |= cudaDeviceSynchronize() != cudaSuccess;
  int err = 1;
  cudaMemcpy(&err, derr, 4, cudaMemcpyDeviceToHost);
  cudaMemcpy(order, dorder, n * 4, cudaMemcpyDeviceToHost);
  cudaMemcpy(n_before, dn, n, cudaMemcpyDeviceToHost);
  pin::Sort s;
  const char* at = scratch + n * 16 + pin::status_bytes(n);  // as fragment_order places it
  at = reinterpret_cast<const char*>((reinterpret_cast<uintptr_t>(at) + 255) & ~(uintptr_t)255);
  cudaMemcpy(&s, at, sizeof(s), cudaMemcpyDeviceToHost);
  *width = s.width;
  cudaFree(dF); cudaFree(dorder); cudaFree(derr); cudaFree(dn); cudaFree(scratch);
  return rc || err ? -1 : s.passes;
}
