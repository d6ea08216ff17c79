// Seeded initial conditions generated on the device (pin_set_ic_seed): the
// same counter-based generator as the host module (include/pin_ic.h: P(k) =
// A k^ns T_BBKS(k/Gamma)^2, splitmix64 keyed on (seed, linear mode index),
// Box-Muller, Hermitian symmetry on the kz = 0 and kz = N/2 planes), each mode
// computed independently in FP64 with the device's own math functions and
// cast to FP32.  It produces inputs only, none of the collapse arithmetic.
#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.cuh"

namespace pin {
namespace {

constexpr uint64_t kGolden = 0x9E3779B97F4A7C15ULL;

__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  uint64_t z = x + kGolden;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

__device__ __forceinline__ double bbks(double q) {
  if (q <= 0.0) return 1.0;
  const double a = 2.34 * q;
  const double lead = log(1.0 + a) / a;
  // explicit rounded product: no fused multiply-add, as in the host build
  const double p = 1.0 + __dmul_rn(3.89, q) + pow(16.1 * q, 2.0) + pow(5.46 * q, 3.0) + pow(6.71 * q, 4.0);
  return lead * pow(p, -0.25);
}

// sqrt(n^6 P(k) / box^3) of the modes with sx^2 + sy^2 + sz^2 = s2, for every
// s2 up to 3 (n/2)^2 (0 at k = 0).  The spectrum takes five pow and a log per
// evaluation, and a grid has a few hundred modes to every s2.
__global__ void k_ic_scale(int n, double box, double amp, double ns, double gamma, int count, double* tab) {
  for (int s2 = blockIdx.x * blockDim.x + threadIdx.x; s2 < count; s2 += gridDim.x * blockDim.x) {
    const double kk = 2.0 * M_PI / box * sqrt((double)s2);
    double P = 0.0;
    if (kk > 0.0) {
      const double t = bbks(kk / gamma);
      P = amp * pow(kk, ns) * t * t;
    }
    tab[s2] = sqrt((double)n * n * n * (double)n * n * n * P / (box * box * box));
  }
}

// x / sqrt(2), correctly rounded: the quotient by the rounded reciprocal,
// corrected by its exact remainder (Markstein's division; the values here are
// far from the ends of the range).
__device__ __forceinline__ double over_sqrt2(double x) {
  constexpr double d = 1.4142135623730951, inv = 0.70710678118654746;  // RN(sqrt 2), RN(1 / d)
  const double q = x * inv;
  return fma(fma(-q, d, x), inv, q);
}

__device__ __forceinline__ void mode_value(int n, uint64_t key, const double* __restrict__ tab, int ix, int iy, int iz,
                                           double* re, double* im) {
  const int nh = n / 2 + 1;
  const int sx = ix < n / 2 ? ix : ix - n, sy = iy < n / 2 ? iy : iy - n;
  const double scale = __ldg(tab + sx * sx + sy * sy + iz * iz);
  const uint64_t m = ((uint64_t)ix * n + iy) * nh + iz;
  const uint64_t r1 = splitmix64(key + (2 * m + 1) * kGolden);
  const uint64_t r2 = splitmix64(key + (2 * m + 2) * kGolden);
  const double u1 = ((double)((r1 >> 11) + 1)) * 0x1.0p-53;  // (0, 1]
  const double u2 = ((double)(r2 >> 11)) * 0x1.0p-53;        // [0, 1)
  const double rad = sqrt(-2.0 * log(u1));
  double sn, cs;
  sincos(2.0 * M_PI * u2, &sn, &cs);
  *re = over_sqrt2(scale * (rad * cs));
  *im = over_sqrt2(scale * (rad * sn));
}

// One realisation per blockIdx.y; out holds batch half-spectra [n][n][n/2+1].
// Bound by the FP64 pipe (a log, a square root and a sine-cosine pair per
// mode, two lanes per SM and clock): 512^3 75 -> 9.9 ms with the table of
// scales and the two-step division.
__global__ void k_ic_seed(int n, const uint64_t* keys, const double* __restrict__ tab, float2* out) {
  const unsigned nh = n / 2 + 1, un = n;
  const unsigned total = un * un * nh;  // < 2^31: checked at plan creation
  const uint64_t key = keys[blockIdx.y];
  float2* o = out + (size_t)blockIdx.y * total;
  for (unsigned m = blockIdx.x * blockDim.x + threadIdx.x; m < total; m += gridDim.x * blockDim.x) {
    const unsigned r = m / nh;
    const int iz = (int)(m - r * nh);
    const int ix = (int)(r / un), iy = (int)(r % un);
    double re = 0.0, im = 0.0;
    if (m != 0) {
      // the kz = 0 and kz = n/2 planes: the mirror with the lower index is
      // generated, the other one its conjugate
      const bool plane = iz == 0 || iz == n / 2;
      const int jx = (n - ix) % n, jy = (n - iy) % n;
      const unsigned mm = ((unsigned)jx * un + jy) * nh + iz;
      const bool mirror = plane && mm < m;
      mode_value(n, key, tab, mirror ? jx : ix, mirror ? jy : iy, iz, &re, &im);
      if (mirror) im = -im;
      if (plane && mm == m) {
        re *= sqrt(2.0);
        im = 0.0;
      }
    }
    o[m] = make_float2((float)re, (float)im);
  }
}

}  // namespace

size_t ic_table_count(int n) { return (size_t)3 * (n / 2) * (n / 2) + 1; }

cudaError_t generate_ic(int n, double box, const uint64_t* keys_dev, double* table, int batch, double amp, double ns,
                        double gamma, float2* out, cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int count = (int)ic_table_count(n);
  k_ic_scale<<<(unsigned)((count + 127) / 128), 128, 0, st>>>(n, box, amp, ns, gamma, count, table);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const size_t total = (size_t)n * n * (n / 2 + 1);
  const size_t want = (total + 255) / 256;
  const unsigned gx = (unsigned)(want < (size_t)sms * 16 ? want : (size_t)sms * 16);
  k_ic_seed<<<dim3(gx, (unsigned)batch), 256, 0, st>>>(n, keys_dev, table, out);
  return cudaGetLastError();
}

}  // namespace pin
