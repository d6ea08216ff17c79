// pin_collapse_times_noalloc: the collapse-time loop for small grids with no
// device allocation at all, and pin_noalloc_status, which reads back what its
// last call recorded (both declared in include/pin.h).
//
// Who needs it: callers that cannot allocate device memory at call time.  A
// serving process that has already handed the device's memory to its own pool
// has none left for a per-call cudaMalloc; code that runs inside an allocator
// hook must not re-enter the allocator; and a latency-critical caller cannot
// accept cudaFree's implicit device-wide synchronisation.  Such callers pass
// device inputs and outputs, and the workspace (the half-spectra between the
// passes, the per-radius filter tables, the FP64 redo queue, its counters and
// the error word) lives in one file-scope device array below, sized for grids
// up to PIN_NOALLOC_MAX_N.
//
// That array exists once per device and stays allocated on every GPU that
// loads this library until the process exits.  All calls share it and it keeps
// the previous call's contents, so every call rewrites what it reads (tables,
// spectra including their pad columns) and zeroes its counters and error word;
// two calls whose work overlaps on the GPU (different streams, or different
// host threads) race on it and must be serialised by the caller.
//
// The tables are built on the host by the same functions as the plan path's
// (fill_mult, fill_twiddles, padded_half, the redo capacity), staged in a
// file-scope host array and copied in on the caller's stream, and the same
// kernels run with the same launch shapes, so the results equal
// pin_collapse_times bit for bit.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "kernels.cuh"
#include "pin.h"

namespace {

constexpr int kMaxN = PIN_NOALLOC_MAX_N;
constexpr int kMaxScales = 64;
// FP64 redo queue per radius: the plan path's capacity, max(65536, N^3 / 64),
// which is 65536 entries for every N this entry point accepts
constexpr size_t kRedoCap = 65536;
static_assert((size_t)kMaxN * kMaxN * kMaxN / 64 <= kRedoCap, "redo capacity below the plan path's rule");

constexpr size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }
constexpr size_t spec_bytes(int n) { return (size_t)n * n * ((n / 2 + 1 + 3) & ~3) * sizeof(float2); }

// The head of the workspace: {counters, queue counts, error word, the word that
// turns the bands off}, cleared as one by every call.  It lies at the same
// place for every grid, so that pin_noalloc_status reads what the last call to
// have run left there, whichever call was made or captured since.
constexpr size_t kOffCnt = 0;
constexpr size_t kOffRedoCount = kOffCnt + 4 * sizeof(unsigned long long);
constexpr size_t kOffErr = kOffRedoCount + kMaxScales * sizeof(unsigned);
constexpr size_t kOffWide = kOffErr + 8;
constexpr size_t kHeadBytes = align256(kOffWide + 8);

// Where the rest lies for grids of n points a side and groups of `group` radii
// (RadGroup): the running maximum of a group, cleared with the head; Phi0, U
// and V; the tables {twiddles, bands, multipliers}, copied in as one piece; the
// redo queues.
struct Layout {
  int group;
  size_t cap;  // redo entries per radius
  size_t state, phi0, U, V, tw, band, mult, redo, end;
  constexpr Layout(int n, int g) : group(g), cap(), state(), phi0(), U(), V(), tw(), band(), mult(), redo(), end() {
    const size_t n3 = (size_t)n * n * n;
    cap = g > 1 && n3 < kRedoCap ? n3 : kRedoCap;
    state = kHeadBytes;
    phi0 = align256(state + (g > 1 ? n3 * 8 : 0));
    U = phi0 + spec_bytes(n);
    V = U + 3 * spec_bytes(n) * g;
    tw = V + 6 * spec_bytes(n) * g;
    band = tw + (size_t)n * sizeof(float2);
    mult = band + (size_t)kMaxScales * 4 * sizeof(int);
    redo = align256(mult + (size_t)kMaxScales * 3 * n * sizeof(float));
    end = align256(redo + cap * g * sizeof(pin::RedoEntry));
  }
};
// One radius at a time at the largest grid: 13.9 MB; smaller grids use the
// same space for groups of radii (48^3: one, 32^3: five, 16^3: sixteen).
constexpr size_t kScratchBytes = Layout(kMaxN, 1).end;
constexpr int group_of(int n) {
  int g = 1;
  while (g < pin::kMaxGroup && Layout(n, g + 1).end <= kScratchBytes) ++g;
  return g;
}

// The whole device workspace of this entry point (13.9 MB for
// N <= 64).  In host code this name is only a stand-in for the symbol, never
// a device address: the address comes from cudaGetSymbolAddress at set-up.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_setup_mu;
unsigned char* g_scratch_ptr[kMaxDevices] = {};

// Host staging of the tables (filled and copied under g_stage_mu; a copy from
// pageable host memory has consumed its source when cudaMemcpyAsync returns).
std::mutex g_stage_mu;
struct Tables {  // as Layout places them (the twiddles end where the bands begin)
  float2 tw[kMaxN];
  int band[kMaxScales * 4];
  float mult[(size_t)kMaxScales * 3 * kMaxN];
};
Tables g_h_tables;

// Once per device, with that device current: the scratch address, the
// constant twiddle tables and the kernels' shared-memory limits.
pin_status noalloc_setup(int dev, unsigned char** out) {
  std::lock_guard<std::mutex> lk(g_setup_mu);
  if (!g_scratch_ptr[dev]) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || ptr == nullptr) return PIN_ECUDA;
    if (pin::upload_constant_twiddles() != cudaSuccess) return PIN_ECUDA;
    for (int n : {8, 16, 32, 48, 64})
      if (pin::prepare_kernels(n) != cudaSuccess) return PIN_ECUDA;
    g_scratch_ptr[dev] = static_cast<unsigned char*>(ptr);
  }
  *out = g_scratch_ptr[dev];
  return PIN_OK;
}

int current_device() {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return -1;
  return dev;
}

}  // namespace

extern "C" pin_status pin_collapse_times_noalloc(const void* delta_k, int dtype, int n, double box,
                                                 int nscales, const double* radii, int correction,
                                                 float* F_max, int32_t* scale_idx, void* stream) {
  if (!delta_k || !radii || !F_max || !scale_idx) return PIN_EINVAL;
  if (n > kMaxN || n < 8 || !pin::size_supported(n)) return PIN_EINVAL;  // beyond the static workspace
  if (dtype != PIN_C64 && dtype != PIN_C128) return PIN_EINVAL;
  if (nscales < 1 || nscales > kMaxScales || !(box > 0.0) || !std::isfinite(box)) return PIN_EINVAL;
  if (correction != PIN_CORR_NONE && correction != PIN_CORR_SPHERE) return PIN_EINVAL;
  for (int s = 0; s < nscales; ++s)
    if (!(radii[s] >= 0.0) || !std::isfinite(radii[s])) return PIN_EINVAL;
  const int dev = current_device();
  if (dev < 0) return PIN_ECUDA;
  unsigned char* base = nullptr;
  pin_status st = noalloc_setup(dev, &base);
  if (st != PIN_OK) return st;

  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  const pin::PassShape sh = pin::pass_shape(n);
  const int nhp = pin::padded_half(n);
  const size_t spec = (size_t)n * n * nhp;
  const Layout at(n, group_of(n));
  float2* phi0 = reinterpret_cast<float2*>(base + at.phi0);
  float2* U = reinterpret_cast<float2*>(base + at.U);
  float2* V = reinterpret_cast<float2*>(base + at.V);
  unsigned long long* state = at.group > 1 ? reinterpret_cast<unsigned long long*>(base + at.state) : nullptr;
  float* mult = reinterpret_cast<float*>(base + at.mult);
  float2* tw = reinterpret_cast<float2*>(base + at.tw);
  unsigned long long* cnt = reinterpret_cast<unsigned long long*>(base + kOffCnt);
  unsigned* redo_count = reinterpret_cast<unsigned*>(base + kOffRedoCount);
  int* err = reinterpret_cast<int*>(base + kOffErr);
  int* band = reinterpret_cast<int*>(base + at.band);
  int* wide = reinterpret_cast<int*>(base + kOffWide);
  pin::RedoEntry* redo_list = reinterpret_cast<pin::RedoEntry*>(base + at.redo);
  CUtensorMap tm_x[2], tm_y[2];  // staged and whole-line boxes
  const int tc = sh.tc;  // the default tile width, as a new plan runs
  for (int m = 0; m < 2; ++m) {
    const int boxes = m ? pin::store_boxes(n) : pin::stage_boxes(sh.E);
    if (pin::make_tmap_x(&tm_x[m], phi0, n, n, nhp, 1, tc, boxes) != cudaSuccess ||
        pin::make_tmap_y(&tm_y[m], U, n, n, nhp, spec, 3 * at.group, 1, tc, boxes) != cudaSuccess)
      return PIN_ECUDA;
  }
  const double dcorr = pin::correction_dcorr();
  const size_t n3 = (size_t)n * n * n;
  {
    // per radius [3][n] multipliers (cubic grid: one table serves all axes)
    std::lock_guard<std::mutex> lk(g_stage_mu);
    float2* h_tw = g_h_tables.tw + (kMaxN - n);
    for (int s = 0; s < nscales; ++s) {
      float* m = g_h_tables.mult + (size_t)s * 3 * n;
      pin::fill_mult(m, n, box, radii[s]);
      pin::fill_band(g_h_tables.band + 4 * s, m, n, m, n, m, n, nhp);
    }
    pin::fill_twiddles(h_tw, n, sh);
    if (cudaMemcpyAsync(tw, h_tw, at.mult - at.tw + (size_t)nscales * 3 * n * sizeof(float), cudaMemcpyHostToDevice,
                        cs) != cudaSuccess)
      return PIN_ECUDA;
  }
  if (cudaMemsetAsync(cnt, 0, kHeadBytes + (state ? n3 * sizeof(*state) : 0), cs) != cudaSuccess ||
      pin::launch_load_phi0(delta_k, dtype, n, n, n, nhp, box, 1, phi0, wide, cs) != cudaSuccess ||
      (!state && (cudaMemsetAsync(F_max, 0, n3 * sizeof(float), cs) != cudaSuccess ||
                  cudaMemsetAsync(scale_idx, 0xFF, n3 * sizeof(int32_t), cs) != cudaSuccess)))
    return PIN_ECUDA;

  static const int vout[6] = {0, 3, 4, 1, 2, 5};
  static const int sel[6] = {2, 1, 1, 0, 0, 0};
  static const int ym[6] = {0, 1, 0, 2, 0, 1};
  static const int zm[6] = {0, 0, 1, 0, 2, 1};
  // the plan path's order: ascending radius, equal radii by index
  int order[kMaxScales];
  for (int s = 0; s < nscales; ++s) order[s] = s;
  std::stable_sort(order, order + nscales, [&](int a, int b) { return radii[a] < radii[b]; });
  for (int k = 0; k < nscales; k += at.group) {
    const int s = order[k];
    pin::RadGroup rad{};
    rad.n = std::min(at.group, nscales - k);
    rad.mult_set = 3 * n;
    for (int g = 0; g < rad.n; ++g) {
      rad.ms[g] = order[k + g];
      rad.prev[g] = k + g >= at.group ? order[k + g - at.group] : -1;
    }
    rad.band = band;
    rad.wide = wide;
    pin::ArgsX ax{};
    ax.tm = tm_x[0];
    ax.tm_full = tm_x[1];
    ax.src = phi0;
    for (int f = 0; f < 3; ++f) { ax.dst[f] = U + f * spec; ax.xm[f] = f; }
    ax.nout = 3;
    ax.ny = n;
    ax.mult = mult;
    ax.rad = rad;
    ax.tw = tw;
    ax.nhp = nhp;
    ax.col_unit = tc;
    ax.batch = 1;
    ax.err = err;
    pin::ArgsY ay{};
    ay.tm = tm_y[0];
    ay.tm_full = tm_y[1];
    for (int f = 0; f < 3; ++f) ay.src[f] = U + f * spec;
    for (int o = 0; o < 6; ++o) {
      ay.dst[o] = V + vout[o] * spec;
      ay.sel[o] = sel[o];
      ay.ym[o] = ym[o];
      ay.zm[o] = zm[o];
      ay.muli[o] = 0;
    }
    ay.nout = 6;
    ay.nx = n;
    ay.nz = n;
    ay.mult = mult;
    ay.mult_z = mult;
    ay.rad = rad;
    ay.tw = tw;
    ay.nhp = nhp;
    ay.batch = 1;
    ay.err = err;
    pin::ArgsZ az{};
    for (int f = 0; f < 6; ++f) az.src[f] = V + f * spec;
    az.nfields = 6;
    az.nlines = n * n;
    az.npart = n * n * n;
    az.tw = tw;
    az.nhp = nhp;
    az.fmax = F_max;
    az.idx = scale_idx;
    az.scale = s;
    if (state) {
      az.state = state;
      az.nrad = rad.n;
      for (int g = 0; g < rad.n; ++g) az.ms[g] = rad.ms[g];
      az.gstride = 6 * spec;
    }
    az.correction = correction;
    az.dcorr_d = dcorr;
    az.dcorr_f = (float)dcorr;
    az.tau_eig = 2e-4f;
    az.tau_root = 1e-3f;
    az.counters = cnt;
    az.redo_list = redo_list;
    az.redo_count = redo_count + k;
    az.redo_cap = (unsigned)at.cap;
    if (pin::launch_x(n, tc, 0, ax, cs) != cudaSuccess || pin::launch_y(n, tc, 0, ay, cs) != cudaSuccess ||
        pin::launch_z(n, az, false, cs) != cudaSuccess ||
        pin::launch_redo(az, cs) != cudaSuccess)
      return PIN_ECUDA;
  }
  if (state && pin::launch_unpack(state, n3, F_max, scale_idx, cs) != cudaSuccess) return PIN_ECUDA;
  return PIN_OK;
}

extern "C" pin_status pin_noalloc_status(int* wait_failed, uint64_t* counters3) {
  if (!wait_failed || !counters3) return PIN_EINVAL;
  const int dev = current_device();
  if (dev < 0) return PIN_ECUDA;
  unsigned char* base = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_setup_mu);
    base = g_scratch_ptr[dev];
  }
  if (!base) return PIN_ESTATE;  // no call has run on this device
  unsigned long long c[3] = {0, 0, 0};
  int e = 0;
  if (cudaMemcpy(c, base + kOffCnt, sizeof(c), cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemcpy(&e, base + kOffErr, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
    return PIN_ECUDA;
  *wait_failed = e != 0;
  for (int i = 0; i < 3; ++i) counters3[i] = c[i];
  return e ? PIN_ECUDA : PIN_OK;
}
