// Launch interface of the collapse-time passes (kernels.cu).
//
// Spectral arrays are half-spectra stored [kx][ky][kz] with kz padded to an
// even stride NHP >= N/2+1 (pad modes are zero), complex64.  The filtered
// Hessian spectrum of Sec. 2.1.1,
//   T_ij(k) = (k_i k_j / k^2) W(kR) delta(k),
// is separable once Phi0 = delta / k^2 is formed (once per field):
//   T_ij = mx(kx) my(ky) mz(kz) Phi0,   m in {W, k W, k^2 W} per axis
// (W = exp(-k^2 R^2/2) = Wx Wy Wz, and k carries a zero on the Nyquist index
// for the odd multipliers), so the x pass needs three transforms and only the
// y and z passes carry all six components.
#pragma once
#include <cuda.h>  // CUtensorMap (the encoder itself is fetched from the driver at run time)
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace pin {

constexpr int kMaxFields = 9;

// The error word of a plan (and of the allocation-free entry point): what gave
// up a bounded wait since the host last read it.
enum { kErrNone = 0, kErrTransfer = 1, kErrOrder = 2 };

// Filter support.  W = exp(-k^2 R^2 / 2) underflows: past about kR = 14 the
// FP32 axis factors {W, k W, k^2 W} / n are exactly zero, and with them every
// product and every line they multiply.  At 768^3 with 4 Mpc/h cells and 40
// radii from 120 to 4 Mpc/h, 55 % of the radii have such modes, and 30 % of
// all z columns, 41 % of all (ky, kz) lines are zero.  A band holds, per
// radius, the largest |wavenumber index| with a non-zero factor of each axis,
// {x, y, z, 0}; the x and y passes neither load nor transform what lies
// outside (per radius of such a run the x pass takes 0.95 instead of 1.62 ms,
// the y pass, beside the redo, 2.51 instead of 3.35).  The z pass reads whole lines: a test per
// mode costs its issue slots more (3 %) than the loads it saves.  So the
// columns past a radius's z band have to hold zeros in V; the y pass writes
// them where the radius before it in the same buffer (RadGroup::prev) had
// modes, all others are zero already, the radii running from small to large.
// Nothing but exact zeros is left out, so the results are those of the full
// passes: a field with a value that is not finite, or so large that an
// intermediate could overflow (then 0 x inf would make a NaN of a zero), sets
// *wide, and the passes run full.
//
// Radius groups.  A small grid's pass over one radius is a few microseconds of
// work on a part of the SMs, so its launches cover several radii at once: U
// and V hold n sets of spectra back to back, the x and y passes walk the tiles
// of all of them, the z pass has a grid row per radius and keeps its running
// maximum in one 64-bit word per particle.  Lines of at most kGroupMaxN points.
constexpr int kMaxGroup = 16;
constexpr int kGroupMaxN = 128;
struct RadGroup {
  int n;                // radii of this launch (1 where a line has more than kGroupMaxN points)
  int ms[kMaxGroup];    // their multiplier sets
  int prev[kMaxGroup];  // y pass: the set whose spectra the V buffer held before; -1: anything
  int mult_set;         // floats from one set's multipliers to the next
  const int* band;      // {x, y, z, 0} of set 0, sets back to back; null: full
  const int* wide;      // non-zero: full
};
// Band of one radius from the axis factors ([3][n] each).  The z entry of a
// full axis is nhp - 1, so that it covers the pad columns.
void fill_band(int* band4, const float* mx, int nx, const float* my, int ny, const float* mz, int nz, int nhp);
// |Phi0| from which a field runs full: far below where any intermediate of
// the passes can overflow FP32.
float wide_limit(int nx, int ny, int nz, double box);

// x pass (lines of length nx): for each output f, dst[f] = IDFT_x(mult[xm[f]]
// * src).  The source tiles arrive by TMA: tm is a 2D map over src,
// {ny*nhp columns, batch*nx rows} (realisations stacked along rows), box
// {tc, nx/boxes}.
struct ArgsX {
  CUtensorMap tm;       // in stage_boxes, for partial bands
  CUtensorMap tm_full;  // in store_boxes: the fewest, for whole lines
  const float2* src;
  float2* dst[3];
  int xm[3];
  int nout;
  int ny;             // rows of a plane: the columns are (ky, kz), ny * nhp of them
  const float* mult;  // [3][nx] multipliers of set 0 (W, kW, k^2W, each / nx)
  const float2* tw;   // twiddles: w_N^{p k1} [E][P], then w_P^{p1 k2a} [P2][P1] for three levels
  int nhp;
  int batch;          // realisations stacked back to back (same N, radii)
  RadGroup rad;       // radius g's outputs: dst[f] + g * 3 spectra (of all realisations)
  int col_unit;       // the y pass reads the band's columns in tiles of this many: all of them are stored
  int* err;           // set to kErrTransfer if a TMA wait gave up (bounded wait)
  long long wait_cycles;  // budget of a TMA wait in SM clocks; <= 0: the default (2^31)
  CUtensorMap tm_out[3];  // maps of dst[f] (filled at launch when outputs go out by TMA stores)
};

// y pass (lines of length ny): dst[f] = zfac[f](kz) * IDFT_y(mult[ym[f]] *
// src[sel[f]]), where the z factor mult_z[zm[f]](kz), times i when muli[f], is
// constant along a y line.  Outputs are processed in the given order;
// consecutive outputs with the same source share one staged tile.  tm is a 4D
// map over the three source spectra (stored back to back),
// {nhp, ny, batch*nx, 3 per radius}, box {tc, ny/boxes, 1, 1}.
struct ArgsY {
  CUtensorMap tm;       // in stage_boxes, for partial bands
  CUtensorMap tm_full;  // in store_boxes
  const float2* src[3];
  float2* dst[kMaxFields];
  int sel[kMaxFields];
  int ym[kMaxFields];
  int zm[kMaxFields];
  int muli[kMaxFields];
  // optional second store of the same transform with its own z factor
  float2* dst2[kMaxFields];
  int zm2[kMaxFields];
  int muli2[kMaxFields];
  int nout;
  int nx, nz;           // x planes per realisation; z line length (z factors for kz <= nz/2)
  const float* mult;    // [3][ny] y multipliers of set 0
  const float* mult_z;  // [3][nz] z multipliers of set 0
  const float2* tw;
  int nhp;
  int batch;
  RadGroup rad;         // radius g: sources src + g * 3 spectra, outputs dst[o] + g * 6
  int* err;
  long long wait_cycles;
  CUtensorMap tm_out[kMaxFields];  // maps of dst[o] (filled at launch when outputs go out by TMA stores)
};

// A particle whose FP32 collapse is ill-conditioned, finished in FP64 by the
// redo kernel, both kinds queued by the z pass: kind 0 (near-degenerate
// eigenvalue pair) carries the six FP32 Hessian components; kind 1
// (near-tangent or unconverged root) carries the three eigenvalues in
// h[0..2].
struct RedoEntry {
  int q;
  float h[6];
  int kind;
};

// z pass: c2r of each field (its z factor already applied by the y pass),
// then the collapse times and running maximum of every particle, or a dump of
// the real fields.
struct ArgsZ {
  const float2* src[kMaxFields];
  int nfields;
  int nlines;    // batch * N^2 lines along z
  int npart;     // batch * N^3 particles
  int prefetch_blocks;  // z pass: prefetch the lines of block + this many into L2 (0: none)
  const float2* tw;
  int nhp;
  // collapse mode (nfields 6), with the displacement components (nfields 9)
  float* psi_out;   // [3][npart] smoothed displacement of this radius, for queued particles
  float* vstate;    // [3][npart] displacement at R_max, or null
  float* fmax;
  int* idx;
  int scale;
  // radius groups: state != null.  Radius g < nrad (index ms[g]) reads src[f]
  // + g * gstride and queues into redo_list + g * redo_cap, redo_count[g];
  // state[q] = bits of F << 32 | ~index, 0 before any F > 0: its maximum is
  // the larger F and among equal ones the lower index.  fmax, idx, scale unused.
  unsigned long long* state;
  int nrad;
  int ms[kMaxGroup];
  size_t gstride;
  int correction;
  float dcorr_f;
  double dcorr_d;
  float tau_eig;   // FP64 redo when |r| > 1 - tau_eig
  float tau_root;  // FP64 redo when kappa < tau_root
  unsigned long long* counters;  // [0] eigen redo, [1] root redo, [2] list overflow
  RedoEntry* redo_list;          // FP64 redo queue of this radius
  unsigned* redo_count;          // zero before the z pass; one per radius of the call
  unsigned redo_cap;
  // dump mode
  float* out[kMaxFields];
};

struct PassShape {
  int E, P;
  int P1, P2;     // P = P1 * P2; P2 > 1: three-level line transform
  int tc;         // columns per block, x/y passes
  int lines;      // lines per block, z pass
  size_t smem_xy; // dynamic shared bytes, x/y passes
  size_t smem_z;
  int threads_xy, threads_z;
};

// Tensor maps of the x and y passes (host; the encoder comes from the driver
// entry point, so no driver library is linked).  spec_elems is the stride
// between the spectra the y map spans; tc is the tile width (columns) of the
// pass that reads the map, one of xy_tile_options.
// `boxes`: the boxes a tile of rows is moved in (stage_boxes of the pass's
// schedule for loads, store_boxes for stores).
cudaError_t make_tmap_x(CUtensorMap* tm, const float2* src, int nx, int ny, int nhp, int batch, int tc, int boxes);
// 2D map of rows of `cols` complex values (row pitch cols), box {tc, box_rows}
cudaError_t make_tmap_rows(CUtensorMap* tm, const float2* base, int cols, long long rows, int tc, int box_rows);
cudaError_t make_tmap_y(CUtensorMap* tm, const float2* src, int nx, int ny, int nhp, size_t spec_elems, int nspec,
                        int batch, int tc, int boxes);
// Boxes of a staged tile of n rows with E register slots per thread: eighths
// (quarters where E is no multiple of eight), whole slots each, so that a
// band's rows are loaded and a band's slots multiplied without a remainder.
// A TMA box has at most 256 rows, and 768 / 4 rows fit as well.
constexpr int stage_boxes(int E) { return E % 8 == 0 ? 8 : 4; }
constexpr int store_boxes(int n) { return (n + 255) / 256; }
// Radix schedules of the x/y line transforms (fft.cuh ShapeBase<N, V>):
// 0, the default and the z pass's, and 1.
constexpr int kRadixVariants = 2;
// Tile widths the x/y pass over lines of n points can run with radix
// schedule v (opts[0] is the default); returns their number (0 for an
// unsupported size or schedule).
int xy_tile_options(int n, int v, int* opts);

bool size_supported(int n);
PassShape pass_shape(int n);          // schedule 0: z pass, and the x/y defaults
PassShape pass_shape_xy(int n, int v);  // the x/y line transform of schedule v
cudaError_t prepare_kernels(int n);  // sets shared-memory attributes (once per device)
// tc: tile width, one of xy_tile_options(n, v) (anything else runs the
// default of schedule v); v: radix schedule
cudaError_t launch_x(int n, int tc, int v, const ArgsX& a, cudaStream_t st);
cudaError_t launch_y(int n, int tc, int v, const ArgsY& a, cudaStream_t st);
// schedule 1 (kernels_v1.cu)
cudaError_t upload_constant_twiddles_v1();  // that unit's copy of the register-DFT twiddles
cudaError_t prepare_xy_v1(int n);
int xy_tile_options_v1(int n, int* opts);
PassShape pass_shape_xy_v1(int n);
cudaError_t launch_x_v1(int n, int tc, const ArgsX& a, cudaStream_t st);
cudaError_t launch_y_v1(int n, int tc, const ArgsY& a, cudaStream_t st);
cudaError_t launch_z(int n, const ArgsZ& a, bool dump, cudaStream_t st);
// Second-order LPT pieces: the z pass writing the source S of every particle
// (from the six fields in src[0..5]) to out[0]; the inverse-sign transform
// along z of real lines (nlines of them, an even number) into a padded
// half-spectrum; and Phi2 = scale conj(T) / k^2.
cudaError_t launch_z_source(int n, const ArgsZ& a, cudaStream_t st);
cudaError_t launch_fwd_z(int n, const float* src, float2* dst, int nlines, int nhp, const float2* tw,
                         cudaStream_t st);
cudaError_t launch_phi2(const float2* T, float2* out, int nx, int ny, int nz, int nhp, double box, float scale,
                        cudaStream_t st);
// True when lines of n points run three-level transforms.
bool three_level(int n);
// The FP64 redo of every particle the z pass queued (after it, same stream).
cudaError_t launch_redo(const ArgsZ& a, cudaStream_t st);
// state -> F_max and index of every particle (after the last group's redo)
cudaError_t launch_unpack(const unsigned long long* state, size_t n, float* fmax, int* idx, cudaStream_t st);
cudaError_t upload_constant_twiddles();  // per device

// Host helpers shared by the plan path (pin.cu) and the allocation-free entry
// point (noalloc.cu), so that both build identical tables:
//   padded_half      kz stride of the padded half-spectra (n/2 + 1 rounded up
//                    to a multiple of 4 complex values)
//   correction_dcorr 1/delta_c - 1/x3 of the quasi-spherical correction
//   fill_mult        {W, kW, k^2 W} / n of one axis at one radius ([3][n])
//   fill_twiddles    the line transform's twiddles of one axis
//   launch_load_phi0 Phi0 = delta / k^2 into the padded layout (C64 or C128
//                    input, batch realisations back to back); *wide is set to
//                    1 where |Phi0| is not below `limit` (the caller clears it)
int padded_half(int n);
double correction_dcorr();
void fill_mult(float* out, int n, double box, double radius);
void fill_twiddles(float2* t, int n, const PassShape& sh);
cudaError_t launch_load_phi0(const void* src, int dtype, int nx, int ny, int nz, int nhp, double box, int batch,
                             float2* phi0, int* wide, cudaStream_t st);

// All-FP64 loop of a PIN_FP64 plan (fp64.cu): device bytes of its workspace
// (FP64 half-spectrum, twiddles, the tensor, F_max), the input as an FP64
// half-spectrum, the whole radius loop into fmax / idx (N^3 each, running
// maximum from 0 / -1, ties to the lower index; tw: nx + ny + nz values of
// scratch), and the FP32 copy of F_max.
size_t fp64_workspace_bytes(int nx, int ny, int nz);
cudaError_t fp64_load(const void* src, int dtype, int nx, int ny, int nz, double2* d64, cudaStream_t st);
cudaError_t fp64_collapse(const double2* d64, int nx, int ny, int nz, double box, int nscales, const double* radii,
                          int correction, double dcorr, double2* tw, double* h6, double* fmax, int* idx,
                          cudaStream_t st);
cudaError_t fp64_cast(const double* in, size_t n3, float* out, cudaStream_t st);

// Seeded initial conditions on the device (ic_gpu.cu): batch cubic
// half-spectra [n][n][n/2+1] complex64 into out, realisation b keyed by
// keys_dev[b] (the splitmix64 of its seed), amplitude amp of P(k); table is
// scratch for ic_table_count(n) doubles.
size_t ic_table_count(int n);
cudaError_t generate_ic(int n, double box, const uint64_t* keys_dev, double* table, int batch, double amp, double ns,
                        double gamma, float2* out, cudaStream_t st);

// Fragmentation front end (fragment.cu): the particles of one nx*ny*nz grid in
// descending F_max (ties: ascending index) into `order`, and the number of
// their six periodic neighbours that precede them into `n_before`; either
// output may be null.  `scratch` holds fragment_scratch_bytes(N^3) bytes.  A
// block whose wait for an earlier one runs out (wait_cycles as in ArgsX) sets
// *err to kErrOrder.
size_t fragment_scratch_bytes(long n3);
cudaError_t fragment_order(const float* fmax, int nx, int ny, int nz, void* scratch, int32_t* order,
                           uint8_t* n_before, long long wait_cycles, int* err, cudaStream_t st);
int fragment_kernels(bool order, bool counts);  // launches of one fragment_order call

}  // namespace pin
