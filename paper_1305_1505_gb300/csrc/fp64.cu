// All-FP64 collapse-time loop (pin_plan_desc.precision = PIN_FP64): the same
// steps as the FP32 path of Sec. 2.1.1 -- filter the linear field delta(k) at
// each radius, inverse-transform the six components of the deformation tensor,
// eigenvalues and collapse time per grid point, running maximum -- in double
// precision throughout.  It is a debugging and checking mode of the library:
// every other call of a plan runs in FP32.
//
// The FP64 pipe has two lanes per SM and clock, so FP64 operations are what
// the time goes to, and the design is about their number:
//  - two real components ride one complex transform (three full cubes in place
//    of six), filtered as the z lines are loaded, one exponential and one
//    division for a mode and its mirror;
//  - twiddles come from tables;
//  - the x pass keeps its lines of all three cubes in shared memory and goes
//    on to the eigenvalues and collapse times, radii from small to large, and
//    only of particles that can still beat their running maximum: the
//    invariant bound first, then the no-root test, each survivor queued so
//    that the next stage runs on full warps.
// 64^3 x 20 takes 5.4 ms and 128^3 x 10 18.6 ms (38.2 and 97.9 with a transform
// per component, a sincospi per butterfly and every particle solved at every
// radius).
//
// Layout: the half-spectrum d64 [nx][ny][nz/2+1]; three cubes (double2,
// [nx][ny][nz]) in the tensor workspace: xx + i yy, zz + i xy, xz + i yz.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "collapse.cuh"
#include "kernels.cuh"
#include "pin.h"

namespace pin {
namespace {

__device__ __forceinline__ double2 zadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 zsub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 zmuli(double2 a) { return make_double2(-a.y, a.x); }

// delta(k) in the caller's precision -> FP64 half-spectrum
__global__ void k_load64(const void* src, int dtype, size_t count, double2* out) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x) {
    if (dtype == PIN_C64) {
      const float2 v = static_cast<const float2*>(src)[i];
      out[i] = make_double2(v.x, v.y);
    } else {
      out[i] = static_cast<const double2*>(src)[i];
    }
  }
}

// exp(2 pi i j / n) of the three axes, back to back.
__global__ void k_twiddles64(int nx, int ny, int nz, double2* tw) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nx + ny + nz) return;
  const int n = j < nx ? nx : (j < nx + ny ? ny : nz);
  const int k = j < nx ? j : (j < nx + ny ? j - nx : j - nx - ny);
  double sn, cs;
  sincospi(2.0 * (double)k / (double)n, &sn, &cs);
  tw[j] = make_double2(cs, sn);
}

// Inverse transforms X[k] = sum_j x[j] exp(+2 pi i j k / n) (n = 2^a 3^b) of nc
// lines in shared memory, element j of line c at [j * ld + c * cs], through
// tmp (same layout).  Stockham autosort, radix 4, then 2, then 3: at a stage
// of radix r with span Ns, butterfly j takes x[j + t n/r] (t < r), multiplies
// by exp(2 pi i t k / (Ns r)) with k = j mod Ns, applies the length-r DFT and
// writes element (j / Ns) Ns r + k + t Ns; the spans multiply to n.  Returns
// the buffer that holds the result (x or tmp).
__device__ double2* fft64(double2* x, double2* tmp, int n, int nc, int ld, int cs, const double2* __restrict__ tw) {
  int rest = n, Ns = 1;
  while (rest > 1) {
    const int r = (rest % 4 == 0) ? 4 : (rest % 2 == 0 ? 2 : 3);
    const int m = n / r, unit = m / Ns;  // n / (Ns r)
    __syncthreads();
    for (int w = threadIdx.x; w < m * nc; w += blockDim.x) {
      // consecutive threads on consecutive addresses: columns, or one line's points
      const int j = cs == 1 ? w / nc : w % m, c = cs == 1 ? w - j * nc : w / m;
      const int q = j / Ns, k = j - q * Ns;
      const double2* in = x + (size_t)j * ld + (size_t)c * cs;
      double2* out = tmp + (size_t)(q * Ns * r + k) * ld + (size_t)c * cs;
      const int is = m * ld, os = Ns * ld;
      if (r == 4) {
        const double2 v0 = in[0];
        double2 v1 = in[is], v2 = in[2 * is], v3 = in[3 * is];
        if (k) {
          v1 = zmul(v1, __ldg(tw + k * unit));
          v2 = zmul(v2, __ldg(tw + 2 * k * unit));
          v3 = zmul(v3, __ldg(tw + 3 * k * unit));
        }
        const double2 s02 = zadd(v0, v2), d02 = zsub(v0, v2);
        const double2 s13 = zadd(v1, v3), d13 = zmuli(zsub(v1, v3));
        out[0] = zadd(s02, s13);
        out[os] = zadd(d02, d13);
        out[2 * os] = zsub(s02, s13);
        out[3 * os] = zsub(d02, d13);
      } else if (r == 2) {
        const double2 v0 = in[0];
        double2 v1 = in[is];
        if (k) v1 = zmul(v1, __ldg(tw + k * unit));
        out[0] = zadd(v0, v1);
        out[os] = zsub(v0, v1);
      } else {
        // exp(2 pi i / 3) = -1/2 + i sqrt(3)/2
        const double h = 0.86602540378443864676;
        const double2 v0 = in[0];
        double2 v1 = in[is], v2 = in[2 * is];
        if (k) {
          v1 = zmul(v1, __ldg(tw + k * unit));
          v2 = zmul(v2, __ldg(tw + 2 * k * unit));
        }
        const double2 s = zadd(v1, v2), d = zsub(v1, v2);
        const double2 mm = make_double2(v0.x - 0.5 * s.x, v0.y - 0.5 * s.y);
        out[0] = zadd(v0, s);
        out[os] = make_double2(mm.x - h * d.y, mm.y + h * d.x);
        out[2 * os] = make_double2(mm.x + h * d.y, mm.y - h * d.x);
      }
    }
    double2* t = x;
    x = tmp;
    tmp = t;
    Ns *= r;
    rest /= r;
  }
  __syncthreads();
  return x;
}

// z lines: filter and transform.  T_c(k) = (k_i k_j / k^2) W(kR) delta(k) on
// the full line (the half-spectrum's mirror modes as conjugates; k = 0 and,
// for i != j, every mode with k_i or k_j on the Nyquist index zero), paired
// into three complex lines.  Cubic cells: the side along x is `box`, L_y = box
// ny / nx, L_z = box nz / nx.  A block takes nl lines (x, y) of the grid.
__global__ void k_z64(const double2* __restrict__ half, int nx, int ny, int nz, int nl, double box, double radius,
                      const double2* __restrict__ tw, double2* cubes) {
  extern __shared__ double2 zs[];
  const int nh = nz / 2 + 1;
  const size_t n3 = (size_t)nx * ny * nz;
  const double kfx = 2.0 * M_PI / box, kfy = 2.0 * M_PI / (ny == nx ? box : box * ny / nx),
               kfz = 2.0 * M_PI / (nz == nx ? box : box * nz / nx);
  const long long l0 = (long long)blockIdx.x * nl;
  for (int w = threadIdx.x; w < nl * nh; w += blockDim.x) {
    const int l = w / nh, iz = w - l * nh;
    if (l0 + l >= (long long)nx * ny) break;
    const int ix = (int)((l0 + l) / ny), iy = (int)((l0 + l) % ny);
    const int sx = ix < nx / 2 ? ix : ix - nx, sy = iy < ny / 2 ? iy : iy - ny;
    const bool qx = sx == -nx / 2, qy = sy == -ny / 2;
    const double kx = kfx * sx, ky = kfy * sy;
    double2 d = half[((size_t)ix * ny + iy) * nh + iz];
    if (iz == 0 || iz == nz / 2) {
      // the planes that are their own mirror: the Hermitian part, whose
      // transform is the real part of the input's (an input rounded to FP32 is
      // Hermitian there to 1e-8 only, and the paired transform would hand the
      // imaginary part of one component to the other)
      const double2 m = half[((size_t)((nx - ix) % nx) * ny + (ny - iy) % ny) * nh + iz];
      d = make_double2(0.5 * (d.x + m.x), 0.5 * (d.y - m.y));
    }
    const double az = kfz * iz;  // |kz|
    const double k2 = kx * kx + ky * ky + az * az;
    const double g = k2 > 0.0 ? exp(-0.5 * k2 * radius * radius) / k2 : 0.0;
    double2* z = zs + (size_t)l * 3 * nz;
    const bool live = k2 > 0.0;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      // the mode itself (the Nyquist index is -nz/2), then its mirror -kz
      const bool nyq = iz == nz / 2;
      if (side && (iz == 0 || nyq)) break;
      double2 v = d;
      if (side) {
        v = half[((size_t)((nx - ix) % nx) * ny + (ny - iy) % ny) * nh + iz];
        v.y = -v.y;
      }
      const double kz = side || nyq ? -az : az;
      const double mxx = kx * kx * g, myy = ky * ky * g, mzz = kz * kz * g;
      const double mxy = qx || qy ? 0.0 : kx * ky * g, mxz = qx || nyq ? 0.0 : kx * kz * g,
                   myz = qy || nyq ? 0.0 : ky * kz * g;
      const double2 o = make_double2(0.0, 0.0);
      const int at = side ? nz - iz : iz;
      // A + i B of the pair (a, b): (a v.x - b v.y, a v.y + b v.x)
      z[at] = live ? make_double2(mxx * v.x - myy * v.y, mxx * v.y + myy * v.x) : o;
      z[nz + at] = live ? make_double2(mzz * v.x - mxy * v.y, mzz * v.y + mxy * v.x) : o;
      z[2 * nz + at] = live ? make_double2(mxz * v.x - myz * v.y, mxz * v.y + myz * v.x) : o;
    }
  }
  const double2* r = fft64(zs, zs + (size_t)nl * 3 * nz, nz, 3 * nl, 1, nz, tw);
  for (int w = threadIdx.x; w < nl * 3 * nz; w += blockDim.x) {
    const int t = w / nz, l = t / 3;
    if (l0 + l < (long long)nx * ny) cubes[(size_t)(t - 3 * l) * n3 + (size_t)(l0 + l) * nz + (w - t * nz)] = r[w];
  }
}

// y lines of the three cubes in place: tc columns (consecutive z) of one plane
// per block.
__global__ void k_y64(double2* cubes, int ny, int nz, int tc, long long tiles, const double2* __restrict__ tw) {
  extern __shared__ double2 zs[];
  const int ztiles = (nz + tc - 1) / tc;
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
    const long long plane = t / ztiles;  // cube * nx + x
    const int z0 = (int)(t - plane * ztiles) * tc, nc = min(tc, nz - z0);
    double2* base = cubes + plane * ny * nz + z0;
    __syncthreads();
    for (int w = threadIdx.x; w < ny * nc; w += blockDim.x) zs[w] = base[(size_t)(w / nc) * nz + w % nc];
    const double2* r = fft64(zs, zs + (size_t)ny * nc, ny, nc, nc, 1, tw);
    for (int w = threadIdx.x; w < ny * nc; w += blockDim.x) base[(size_t)(w / nc) * nz + w % nc] = r[w];
  }
}

// True when no axis cubic of the coefficients has a real root at or above t by
// more than the rounding of the solver: no_root_from with a margin on the
// critical value, so that a near-tangent root counts as one.
__device__ __forceinline__ bool clear_of_roots(const double c[3], double t) {
  const double gt = ((t - c[0]) * t - c[1]) * t - c[2];
  const double d = c[0] * c[0] + 3.0 * c[1];
  if (!(gt > 0.0)) return false;
  if (d < 0.0) return true;
  const double fs = (c[0] + sqrt(d)) * (1.0 / 3.0);
  const double gs = ((fs - c[0]) * fs - c[1]) * fs - c[2];
  const double size = fabs(fs * fs * fs) + fabs(c[0] * fs * fs) + fabs(c[1] * fs) + fabs(c[2]);
  return fs <= t || gs > 1e-9 * size;
}

// x lines of the three cubes, then eigenvalues, collapse time and running
// maximum (ties of F towards the lower radius index) of their particles: tc
// columns (consecutive (y, z)) per block.
__global__ void k_x64(const double2* __restrict__ cubes, int nx, long long cols, int tc, double norm, int scale,
                      int correction, double dcorr, const double2* __restrict__ tw, double* fmax, int* idx) {
  extern __shared__ double2 zs[];
  __shared__ int s_n[2];
  const size_t n3 = (size_t)nx * cols;
  const long long col0 = (long long)blockIdx.x * tc;
  const int nc = (int)min((long long)tc, cols - col0), np = nx * nc;
  double2* buf[3] = {zs, zs + (size_t)nx * tc, zs + (size_t)2 * nx * tc};
  double2* tmp = zs + (size_t)3 * nx * tc;
  unsigned short* q1 = reinterpret_cast<unsigned short*>(zs + (size_t)4 * nx * tc);
  unsigned short* q2 = q1 + (size_t)nx * tc;
  if (threadIdx.x < 2) s_n[threadIdx.x] = 0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    for (int w = threadIdx.x; w < np; w += blockDim.x)
      buf[c][w] = cubes[(size_t)c * n3 + (size_t)(w / nc) * cols + col0 + w % nc];
    double2* r = fft64(buf[c], tmp, nx, nc, nc, 1, tw);
    if (r == tmp) {
      tmp = buf[c];
      buf[c] = r;
    }
  }
  const CollapseConsts<double> cc{dcorr, correction};
  auto at = [&](int w) { return (size_t)(w / nc) * cols + col0 + w % nc; };
  // the invariant bound
  for (int w = threadIdx.x; w < np; w += blockDim.x) {
    const double2 a = buf[0][w], b = buf[1][w], c = buf[2][w];
    const double h[6] = {a.x * norm, a.y * norm, b.x * norm, b.y * norm, c.x * norm, c.y * norm};
    if (fmax[at(w)] * (1.0 - 1e-9) > collapse_bound<double>(h, cc)) continue;
    q1[atomicAdd(&s_n[0], 1)] = (unsigned short)w;
  }
  __syncthreads();
  // eigenvalues and the no-root test; the survivors' eigenvalues take the
  // place of their tensor
  const int n1 = s_n[0];
  for (int i = threadIdx.x; i < n1; i += blockDim.x) {
    const int w = q1[i];
    const double2 a = buf[0][w], b = buf[1][w], c = buf[2][w];
    const double h[6] = {a.x * norm, a.y * norm, b.x * norm, b.y * norm, c.x * norm, c.y * norm};
    double lam[3];
    eig3<double>(h, lam);
    const double mu1 = lam[0] + lam[1] + lam[2], mu3 = lam[0] * lam[1] * lam[2];
    const double z = 10.0 * (lam[0] - lam[2]) / (mu1 > 0.0 ? mu1 : 1.0);
    const double corr = (correction && mu1 > 0.0) ? mu1 * dcorr * exp(-z * z) : 0.0;
    const double t = (fmax[at(w)] - corr) * (1.0 - 1e-9);
    if (t > 0.0) {
      const double e[3] = {0.5 * lam[0] * (lam[1] + lam[2]), 0.5 * lam[1] * (lam[0] + lam[2]),
                           0.5 * lam[2] * (lam[0] + lam[1])};
      bool clear = true;
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) {
        double co[3];
        axis_coeffs<double>(lam, e, mu3, ax, co);
        clear = clear && clear_of_roots(co, t);
      }
      if (clear) continue;
    }
    buf[0][w] = make_double2(lam[0], lam[1]);
    buf[1][w].x = lam[2];
    q2[atomicAdd(&s_n[1], 1)] = (unsigned short)w;
  }
  __syncthreads();
  const int n2 = s_n[1];
  for (int i = threadIdx.x; i < n2; i += blockDim.x) {
    const int w = q2[i];
    const double lam[3] = {buf[0][w].x, buf[0][w].y, buf[1][w].x};
    double kap;
    const double F = collapse_from_eigs<double>(lam, cc, kap);
    const size_t q = at(w);
    const double fm = fmax[q];
    if (F > fm || (F == fm && F > 0.0 && scale < idx[q])) {
      fmax[q] = F;
      idx[q] = scale;
    }
  }
}

__global__ void k_fill_state64(size_t n3, double* fmax, int* idx) {
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n3; q += (size_t)gridDim.x * blockDim.x) {
    fmax[q] = 0.0;
    idx[q] = -1;
  }
}

__global__ void k_cast64(const double* in, size_t n3, float* out) {
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n3; q += (size_t)gridDim.x * blockDim.x)
    out[q] = (float)in[q];
}

unsigned grid_for(size_t count) { return (unsigned)std::min<size_t>((count + 255) / 256, 152 * 32); }

}  // namespace

size_t fp64_workspace_bytes(int nx, int ny, int nz) {
  const size_t n3 = (size_t)nx * ny * nz, half = (size_t)nx * ny * (nz / 2 + 1);
  return half * 16 + (size_t)(nx + ny + nz) * 16 + 6 * n3 * 8 + n3 * 8;
}

cudaError_t fp64_load(const void* src, int dtype, int nx, int ny, int nz, double2* d64, cudaStream_t st) {
  const size_t count = (size_t)nx * ny * (nz / 2 + 1);
  k_load64<<<grid_for(count), 256, 0, st>>>(src, dtype, count, d64);
  return cudaGetLastError();
}

cudaError_t fp64_collapse(const double2* d64, int nx, int ny, int nz, double box, int nscales, const double* radii,
                          int correction, double dcorr, double2* tw, double* h6, double* fmax, int* idx,
                          cudaStream_t st) {
  const size_t n3 = (size_t)nx * ny * nz;
  const double norm = 1.0 / (double)n3;
  double2* cubes = reinterpret_cast<double2*>(h6);
  const double2 *twx = tw, *twy = tw + nx, *twz = tw + nx + ny;
  // 128-byte rows of columns where the lines leave the shared memory for it
  const int ty = ny <= 384 ? 8 : 4, tx = nx <= 192 ? 8 : 4, nl = std::max(1, 128 / nz);
  const size_t sz = (size_t)nl * 6 * nz * sizeof(double2), sy = (size_t)2 * ny * ty * sizeof(double2),
               sx = (size_t)nx * tx * (4 * sizeof(double2) + 2 * sizeof(unsigned short));
  // the most that any size takes: 73.7, 98.3 and 208.9 KB
  static_assert(768 * 4 * (4 * 16 + 4) + 16 <= 227 * 1024 && 192 * 8 * (4 * 16 + 4) <= 227 * 1024,
                "x lines fit the shared memory");
  cudaError_t e = cudaFuncSetAttribute(k_z64, cudaFuncAttributeMaxDynamicSharedMemorySize, 6 * 768 * 16);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_y64, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * 384 * 8 * 16);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_x64, cudaFuncAttributeMaxDynamicSharedMemorySize, 768 * 4 * 68);
  if (e != cudaSuccess) return e;
  k_fill_state64<<<grid_for(n3), 256, 0, st>>>(n3, fmax, idx);
  k_twiddles64<<<(nx + ny + nz + 127) / 128, 128, 0, st>>>(nx, ny, nz, tw);
  e = cudaGetLastError();
  // from the smallest radius up (equal radii by index), as the FP32 loop runs
  int order[64];
  for (int s = 0; s < nscales; ++s) order[s] = s;
  std::stable_sort(order, order + nscales, [&](int a, int b) { return radii[a] < radii[b]; });
  const long long ytiles = (long long)3 * nx * ((nz + ty - 1) / ty), cols = (long long)ny * nz;
  const unsigned zgrid = (unsigned)(((long long)nx * ny + nl - 1) / nl), xgrid = (unsigned)((cols + tx - 1) / tx);
  const unsigned ygrid = (unsigned)std::min<long long>(ytiles, 1 << 20);
  for (int k = 0; k < nscales && e == cudaSuccess; ++k) {
    const int s = order[k];
    k_z64<<<zgrid, 128, sz, st>>>(d64, nx, ny, nz, nl, box, radii[s], twz, cubes);
    k_y64<<<ygrid, 128, sy, st>>>(cubes, ny, nz, ty, ytiles, twy);
    k_x64<<<xgrid, 256, sx, st>>>(cubes, nx, cols, tx, norm, s, correction, dcorr, twx, fmax, idx);
    e = cudaGetLastError();
  }
  return e;
}

cudaError_t fp64_cast(const double* in, size_t n3, float* out, cudaStream_t st) {
  k_cast64<<<grid_for(n3), 256, 0, st>>>(in, n3, out);
  return cudaGetLastError();
}

}  // namespace pin
