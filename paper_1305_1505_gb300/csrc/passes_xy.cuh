// The x and y passes of the collapse-time loop (Sec. 2.1.1): the filter
// factors of one axis fused into the inverse DFT along that axis, over column
// tiles staged in shared memory by the tensor memory accelerator.  Templated
// on the line length N, the tile width TC and the radix schedule V of the
// line transform (fft.cuh), and included by the two translation units that
// instantiate schedule 0 (kernels.cu) and schedule 1 (kernels_v1.cu).
#pragma once
#include <algorithm>
#include <cstdint>

#include "fft.cuh"
#include "kernels.cuh"

namespace pin {

// ------------------------------------------------------ TMA + mbarrier --
// Source tiles of the x and y passes are brought into shared memory by the
// tensor memory accelerator (cp.async.bulk.tensor), completing on an mbarrier.
// Every wait is bounded (the pass's wait budget, by default 2^31 SM clocks,
// about a second); a block that gives up waits once more, with the full
// default budget, for its copies in flight, reports through the pass's error
// word and returns.

__device__ __forceinline__ uint32_t smem_u32(const void* ptr) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(ptr));
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
constexpr long long kWaitDefault = 1ll << 31;  // SM clocks, about a second at 2 GHz
// try_wait may suspend the thread for a while before it reports "not yet", so
// budgets below kWaitPoll clocks poll with the non-blocking test_wait instead.
constexpr long long kWaitPoll = 1ll << 16;
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity, long long budget) {
  const long long t0 = clock64();
  if (budget < kWaitPoll) {
    while (!mbar_test_wait(bar, parity))
      if (clock64() - t0 > budget) return false;
    return true;
  }
  while (!mbar_try_wait(bar, parity))
    if (clock64() - t0 > budget) return false;
  return true;
}
// Block-uniform wait: true when the staged tile has landed for every thread.
// budget <= 0 selects the default.  On a timeout the block waits once more,
// with the default budget, for its copies in flight (so that no block exits
// with a transfer pending), records the error and the caller returns.
__device__ __forceinline__ bool stage_ready(uint32_t bar, uint32_t parity, int* err, long long budget) {
  const bool ok = mbar_wait_bounded(bar, parity, budget > 0 ? budget : kWaitDefault);
  if (__syncthreads_and(ok)) return true;
  mbar_wait_bounded(bar, parity, kWaitDefault);
  if (threadIdx.x == 0) atomicExch(err, kErrTransfer);
  return false;
}
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* tm, int c0, int c1,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* tm, int c0, int c1, uint32_t src) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
               ::"l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(src)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* tm, int c0, int c1, int c2,
                                            int c3, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
      : "memory");
}

// Staged-tile geometry of a line: kBoxes boxes of kRows rows, kSlots register
// slots each.
template <int N, int V> struct Stage {
  static constexpr int kBoxes = stage_boxes(Shape<N, V>::E);
  static constexpr int kRows = N / kBoxes;
  static constexpr int kSlots = Shape<N, V>::E / kBoxes;
  static_assert(kRows <= 256 && kSlots * kBoxes == Shape<N, V>::E, "boxes hold whole slots");
};
template <int N> struct Store {
  static constexpr int kBoxes = store_boxes(N);
  static constexpr int kRows = N / kBoxes;
};

// The boxes that hold rows |index| <= b of a line of N points: [0, lo) and
// [hi, kBoxes).  part: some row of the line lies outside.
struct BoxRange {
  int lo, hi;
  bool part;
  __device__ __forceinline__ bool has(int box) const { return box < lo || box >= hi; }
  __device__ __forceinline__ bool edge(int box) const { return part && (box == lo - 1 || box == hi); }
  __device__ __forceinline__ int count(int boxes) const { return min(boxes, lo + boxes - hi); }
};
template <int N, int V>
__device__ __forceinline__ BoxRange boxes_of(int b) {
  using G = Stage<N, V>;
  if (2 * b + 1 >= N) return BoxRange{G::kBoxes, G::kBoxes, false};
  return BoxRange{b / G::kRows + 1, (N - b) / G::kRows, true};
}

// Outputs of the x pass, and of the y pass in single-store mode, go out by
// TMA bulk tensor stores of the output tile (written into the exchange
// buffer in tile order) instead of per-thread stores: the warps leave the
// global store queue to the copy engine (x 1.80 -> 1.62 ms, y 3.58 -> 3.36
// ms per radius at 768^3).
// Three-level lines hold half the registers per thread: the z pass is sized
// for more resident blocks (one line per block, 96 threads, nine blocks per
// SM at 72 registers: measured against four 192-thread blocks at 80
// registers, 768^3 z pass 5.21 -> 4.90 ms per radius); with the velocity
// fields (five transforms per line, 160 threads) five blocks (384^3 x 10: three
// 17.4, four 15.5, five 14.8, six 15.3 ms a call).
#ifndef PIN_Z_MINB3
#define PIN_Z_MINB3 9
#endif
#ifndef PIN_Z_MINB3V
#define PIN_Z_MINB3V 5
#endif
template <int N, int TC = 16, int V = 0> struct MinBlocks {
  using S = Shape<N, V>;
  // three-level x/y blocks (TC columns x P threads) are sized for 512
  // resident threads per SM; two-level ones for as many blocks as their
  // shared memory (staged tile, exchange, tables) lets an SM hold, as long as
  // that leaves a thread registers for its E values and a transform's
  // temporaries (4 E + 24: uncapped, the band's cases take a third more and
  // cost the 256^3 y pass a block per SM, 110 -> 131 us)
  static constexpr int kSmem = 2 * N * TC * 8 + S::kTw * 8 + 12 * N + 1280;
  static constexpr int kByRegs = 65536 / (TC * S::P * ((4 * S::E + 24 + 7) / 8 * 8));
  static constexpr int kBySmem = (227 * 1024) / kSmem;
  static constexpr int kMin = kBySmem < kByRegs ? kBySmem : kByRegs;
  static constexpr int kTwo = kMin < 24 ? kMin : 24;  // an SM holds at most 32 blocks
  static constexpr int xy = S::P2 > 1 ? 512 / (TC * S::P) : (kTwo > 1 ? kTwo : 1);
  static constexpr int z = Shape<N>::P2 > 1 ? PIN_Z_MINB3 : (Shape<N>::E <= 16 ? 6 : 8);
  static constexpr int zv = Shape<N>::P2 > 1 ? PIN_Z_MINB3V : (Shape<N>::E <= 16 ? 6 : 4);
  // the dump and source modes only transform: no cap at the two-level sizes
  // (192- or 96-thread blocks, at least two or four to an SM at 512)
  static constexpr int zt = Shape<N>::P2 > 1 ? PIN_Z_MINB3 : (N >= 384 ? 4 : 1);
};

// Slots of a staged tile times their axis factors; slots outside the band are
// zero (their boxes are not loaded).  GUARD: rows of the band's edge boxes
// that lie outside the band hold whatever an earlier radius or field left
// there (the x pass stores only the band's ky rows), so they are set to zero
// instead of being multiplied by their zero factor.
template <int N, int TC, int V, bool GUARD>
__device__ __forceinline__ void load_slots(float2 (&v)[Shape<N, V>::E], const float2* s_st, const float* mt,
                                           const BoxRange& rows, int b0, int p, int c) {
  using G = Stage<N, V>;
  constexpr int E = Shape<N, V>::E, P = Shape<N, V>::P;
  if (!rows.part) {
#pragma unroll
    for (int t = 0; t < E; ++t) v[t] = cscale(s_st[(p + P * t) * TC + c], mt[P * t]);
    return;
  }
#pragma unroll
  for (int b = 0; b < G::kBoxes; ++b) {
    const bool in = rows.has(b), edge = GUARD && rows.edge(b);
#pragma unroll
    for (int i = 0; i < G::kSlots; ++i) {
      const int t = b * G::kSlots + i, n = p + P * t;
      v[t] = make_float2(0.f, 0.f);
      if (in && !(edge && n > b0 && n < N - b0)) v[t] = cscale(s_st[n * TC + c], mt[P * t]);
    }
  }
}

// Lines short enough for radius groups (RadGroup).
template <int N> constexpr bool kMultiRad = N <= kGroupMaxN;

// Walk over the x pass's tiles: radius by radius, realisation by realisation,
// the columns of the filter's support: ky rows 0..by and ny-by..ny-1, columns
// kz < ncz (the y pass's tiles are read whole).  A full plane is walked as one
// run of columns; a partial one row by row, ktiles tiles to a row (the last
// may run past the row's end: it then computes the first columns of the next
// row as well, which come out the same from every tile that holds them).
template <int N, int TC, int V>
struct WalkX {
  int g, base;     // radius of the launch, its first tile
  int by, nrows, ktiles, tpr, ntiles;  // tiles of a realisation and of the radius; the last may run past the columns
  bool flat;
  BoxRange rows;   // kx boxes
  __device__ __forceinline__ explicit WalkX(const ArgsX& a) : g(0), base(0) { init(a); }
  __device__ __forceinline__ void init(const ArgsX& a) {
    const int* b = a.rad.band ? a.rad.band + 4 * a.rad.ms[g] : nullptr;
    const bool part = b != nullptr && __ldg(a.rad.wide) == 0;
    by = part ? __ldg(b + 1) : a.ny / 2;
    const int ncz = part ? min(a.nhp, (__ldg(b + 2) / a.col_unit + 1) * a.col_unit) : a.nhp;
    rows = boxes_of<N, V>(part ? __ldg(b) : N / 2);
    flat = 2 * by + 1 >= a.ny && ncz >= a.nhp;
    nrows = min(a.ny, 2 * by + 1);
    ktiles = (ncz + TC - 1) / TC;
    tpr = flat ? (a.ny * a.nhp + TC - 1) / TC : nrows * ktiles;
    ntiles = tpr * a.batch;
  }
  // to the radius of `tile` (not before the current one); false past the last
  __device__ __forceinline__ bool seek(const ArgsX& a, int tile) {
    if constexpr (kMultiRad<N>) {
      while (tile >= base + ntiles) {
        if (g + 1 >= a.rad.n) return false;
        base += ntiles;
        ++g;
        init(a);
      }
      return true;
    } else {
      return tile < ntiles;
    }
  }
  __device__ __forceinline__ int col(const ArgsX& a, int t) const {  // first column of tile t of a realisation
    if (flat) return t * TC;
    const int row = t / ktiles;
    return (row <= by ? row : a.ny - nrows + row) * a.nhp + (t - row * ktiles) * TC;
  }
};

// The same for the y pass: radius by radius, plane by plane, columns kz <= bz.
template <int N, int TC, int V>
struct WalkY {
  int g, base, by, ktiles, ntiles;
  BoxRange rows;  // ky boxes
  __device__ __forceinline__ explicit WalkY(const ArgsY& a) : g(0), base(0) { init(a); }
  __device__ __forceinline__ void init(const ArgsY& a) {
    const int* b = a.rad.band ? a.rad.band + 4 * a.rad.ms[g] : nullptr;
    const bool part = b != nullptr && __ldg(a.rad.wide) == 0;
    by = part ? __ldg(b + 1) : N / 2;
    rows = boxes_of<N, V>(by);
    ktiles = ((part ? __ldg(b + 2) + 1 : a.nhp) + TC - 1) / TC;
    ntiles = a.nx * a.batch * ktiles;
  }
  __device__ __forceinline__ bool seek(const ArgsY& a, int tile) {
    if constexpr (kMultiRad<N>) {
      while (tile >= base + ntiles) {
        if (g + 1 >= a.rad.n) return false;
        base += ntiles;
        ++g;
        init(a);
      }
      return true;
    } else {
      return tile < ntiles;
    }
  }
};

// ---------------------------------------------------------------- x pass --
// Lines along x: column index col in [0, N*nhp) enumerates (ky, kz); element
// (kx, col) sits at kx*N*nhp + col, so a row of TC columns is contiguous.  A
// persistent block walks column tiles; the staged Phi0 tile serves all
// outputs, and the next tile is requested as soon as the last output has read
// the current one into registers.  Each output tile leaves by TMA stores
// (columns past the last are clipped by the map).
template <int N, int TC, int V>
__global__ void __launch_bounds__(TC* Shape<N, V>::P, MinBlocks<N, TC, V>::xy)
    k_pass_x(const __grid_constant__ ArgsX a) {
  constexpr int E = Shape<N, V>::E, P = Shape<N, V>::P, NTW = Shape<N, V>::kTw;
  using L = XLayoutCols<E, P, TC, Shape<N, V>::P1>;
  using G = Stage<N, V>;
  using GS = Store<N>;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  // staged tile [N][TC]; TMA destinations start on a 128-byte boundary
  float2* s_st = reinterpret_cast<float2*>(smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127));
  float2* s_x = s_st + N * TC;
  float2* s_tw = s_x + L::kSize;
  float* s_m = reinterpret_cast<float*>(s_tw + NTW);  // [3][N] multipliers
  __shared__ __align__(8) unsigned long long s_bar;
  __shared__ int s_xm[3];
  const int tid = threadIdx.x, c = tid % TC, p = tid / TC;
  const uint32_t bar = smem_u32(&s_bar);
  for (int i = tid; i < NTW; i += TC * P) s_tw[i] = a.tw[i];
  int g_m = 0;  // radius whose multipliers s_m holds
  for (int i = tid; i < 3 * N; i += TC * P) s_m[i] = a.mult[(size_t)a.rad.ms[0] * a.rad.mult_set + i];
  if (tid < 3) s_xm[tid] = a.xm[tid];
  if (tid == 0) {
    mbar_init(bar, 1);
    mbar_init_fence();
  }
  __syncthreads();
  WalkX<N, TC, V> cur(a);
  WalkX<N, TC, V> nxt = cur;
  auto issue = [&](const WalkX<N, TC, V>& w, int tile) {
    const int t = tile - w.base, r = t / w.tpr, c0 = w.col(a, t % w.tpr);
    mbar_expect_tx(bar, w.rows.count(G::kBoxes) * G::kRows * TC * 8);
    if (!w.rows.part) {
#pragma unroll
      for (int b = 0; b < GS::kBoxes; ++b)
        tma_load_2d(smem_u32(s_st + b * GS::kRows * TC), &a.tm_full, c0, r * N + b * GS::kRows, bar);
      return;
    }
#pragma unroll
    for (int b = 0; b < G::kBoxes; ++b)
      if (w.rows.has(b)) tma_load_2d(smem_u32(s_st + b * G::kRows * TC), &a.tm, c0, r * N + b * G::kRows, bar);
  };
  if (tid == 0 && nxt.seek(a, blockIdx.x)) issue(nxt, blockIdx.x);
  uint32_t parity = 0;
  // TMA stores: an output tile is written into the exchange buffer in tile
  // order and stored by the copy engine; the next transform's first
  // exchange waits (in the hook) until the engine has read it
  bool pending = false;
  auto wait_store = [&] {
    if (pending) {
      if (tid == 0) bulk_wait_read();
      __syncthreads();
      pending = false;
    }
  };
  for (int tile = blockIdx.x; cur.seek(a, tile); tile += gridDim.x) {
    if (!stage_ready(bar, parity, a.err, a.wait_cycles)) {
      if (tid == 0) bulk_wait_all();
      return;
    }
    parity ^= 1;
    if (kMultiRad<N> && cur.g != g_m) {  // every thread is past its last read of s_m
      g_m = cur.g;
      for (int i = tid; i < 3 * N; i += TC * P) s_m[i] = a.mult[(size_t)a.rad.ms[g_m] * a.rad.mult_set + i];
      __syncthreads();
    }
    const int tt = tile - cur.base;
    const int col0 = cur.col(a, tt % cur.tpr), row0 = (tt / cur.tpr + cur.g * 3 * a.batch) * N;
    const BoxRange rows = cur.rows;
#pragma unroll 1
    for (int f = 0; f < a.nout; ++f) {
      const float* mt = s_m + s_xm[f] * N + p;
      float2 v[E];
      load_slots<N, TC, V, false>(v, s_st, mt, rows, 0, p, c);
      if (f == a.nout - 1) {
        __syncthreads();  // the tile has been read by every thread
        if (tid == 0 && nxt.seek(a, tile + gridDim.x)) {
          fence_proxy_async();
          issue(nxt, tile + gridDim.x);
        }
      }
      fft_line<N, L, false, V>(v, p, c, s_x, s_tw, wait_store);
      __syncthreads();  // every thread has read its last exchange values
#pragma unroll
      for (int j = 0; j < E; ++j) s_x[fft_out_index<N, V>(p, j) * TC + c] = v[j];
      fence_proxy_async();
      __syncthreads();
      if (tid == 0) {
#pragma unroll
        for (int b = 0; b < GS::kBoxes; ++b)
          tma_store_2d(&a.tm_out[f], col0, row0 + b * GS::kRows, smem_u32(s_x + b * GS::kRows * TC));
        bulk_commit();
      }
      pending = true;
    }
  }
  if (tid == 0) bulk_wait_all();
}

// ---------------------------------------------------------------- y pass --
// Lines along y: a tile is TC consecutive kz of one x plane; element
// (ky, kz) of plane x sits at (x*N + ky)*nhp + kz.  Columns past nhp are
// zero-filled by the tensor map and not stored.  Without second stores each
// output tile leaves by TMA stores; with them (DUAL) by per-thread stores.
template <int N, int TC, bool DUAL, int V>
__global__ void __launch_bounds__(TC* Shape<N, V>::P, MinBlocks<N, TC, V>::xy)
    k_pass_y(const __grid_constant__ ArgsY a) {
  constexpr int E = Shape<N, V>::E, P = Shape<N, V>::P, NTW = Shape<N, V>::kTw;
  using L = XLayoutCols<E, P, TC, Shape<N, V>::P1>;
  using G = Stage<N, V>;
  using GS = Store<N>;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float2* s_st = reinterpret_cast<float2*>(smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127));
  float2* s_x = s_st + N * TC;
  float2* s_tw = s_x + L::kSize;
  float* s_m = reinterpret_cast<float*>(s_tw + NTW);
  __shared__ __align__(8) unsigned long long s_bar;
  __shared__ float2* s_dst[kMaxFields];
  __shared__ float2* s_dst2[kMaxFields];
  __shared__ int s_sel[kMaxFields], s_ym[kMaxFields], s_zm[kMaxFields], s_mi[kMaxFields];
  __shared__ int s_zm2[kMaxFields], s_mi2[kMaxFields];
  const int tid = threadIdx.x, c = tid % TC, p = tid / TC;
  const uint32_t bar = smem_u32(&s_bar);
  for (int i = tid; i < NTW; i += TC * P) s_tw[i] = a.tw[i];
  int g_m = 0;  // radius whose multipliers s_m holds
  for (int i = tid; i < 3 * N; i += TC * P) s_m[i] = a.mult[(size_t)a.rad.ms[0] * a.rad.mult_set + i];
  if (tid < kMaxFields) {
    s_dst[tid] = a.dst[tid];
    s_sel[tid] = a.sel[tid] < 3 ? a.sel[tid] : 0;
    s_ym[tid] = a.ym[tid];
    s_zm[tid] = a.zm[tid];
    s_mi[tid] = a.muli[tid];
    s_dst2[tid] = a.dst2[tid];
    s_zm2[tid] = a.zm2[tid];
    s_mi2[tid] = a.muli2[tid];
  }
  if (tid == 0) {
    mbar_init(bar, 1);
    mbar_init_fence();
  }
  __syncthreads();
  const int nhp = a.nhp, nout = a.nout;
  WalkY<N, TC, V> cur(a);
  WalkY<N, TC, V> nxt = cur;
  auto issue = [&](const WalkY<N, TC, V>& w, int tile, int src) {
    const int t = tile - w.base, x = t / w.ktiles, kz0 = (t - x * w.ktiles) * TC, sp = src + 3 * w.g;
    mbar_expect_tx(bar, w.rows.count(G::kBoxes) * G::kRows * TC * 8);
    if (!w.rows.part) {
#pragma unroll
      for (int b = 0; b < GS::kBoxes; ++b)
        tma_load_4d(smem_u32(s_st + b * GS::kRows * TC), &a.tm_full, kz0, b * GS::kRows, x, sp, bar);
      return;
    }
#pragma unroll
    for (int b = 0; b < G::kBoxes; ++b)
      if (w.rows.has(b)) tma_load_4d(smem_u32(s_st + b * G::kRows * TC), &a.tm, kz0, b * G::kRows, x, sp, bar);
  };
  if (tid == 0 && nxt.seek(a, blockIdx.x)) issue(nxt, blockIdx.x, s_sel[0]);
  uint32_t parity = 0;
  // TMA stores (single-store mode): as in the x pass
  constexpr bool kStore = !DUAL;
  bool pending = false;
  auto wait_store = [&] {
    if (kStore && pending) {
      if (tid == 0) bulk_wait_read();
      __syncthreads();
      pending = false;
    }
  };
  for (int tile = blockIdx.x; cur.seek(a, tile); tile += gridDim.x) {
    const int tt = tile - cur.base, x = tt / cur.ktiles, kz0 = (tt - x * cur.ktiles) * TC, kz = kz0 + c;
    const bool ok = kz < nhp;
    const size_t base = (size_t)x * N * nhp + (ok ? kz : 0);
    const float* mult_z = a.mult_z + (size_t)a.rad.ms[cur.g] * a.rad.mult_set;
    const int row0 = (cur.g * 6 * a.nx * a.batch + x) * N;
    const BoxRange rows = cur.rows;
    const int by = cur.by;
#pragma unroll 1
    for (int o = 0; o < nout; ++o) {
      if (o == 0 || s_sel[o] != s_sel[o - 1]) {
        if (!stage_ready(bar, parity, a.err, a.wait_cycles)) {
          if (kStore && tid == 0) bulk_wait_all();
          return;
        }
        parity ^= 1;
        if (kMultiRad<N> && cur.g != g_m) {  // every thread is past its last read of s_m
          g_m = cur.g;
          for (int i = tid; i < 3 * N; i += TC * P) s_m[i] = a.mult[(size_t)a.rad.ms[g_m] * a.rad.mult_set + i];
          __syncthreads();
        }
      }
      const float* mt = s_m + s_ym[o] * N + p;
      float2 v[E];
      load_slots<N, TC, V, true>(v, s_st, mt, rows, by, p, c);
      const bool last_use = (o == nout - 1) || s_sel[o + 1] != s_sel[o];
      if (last_use) {
        __syncthreads();  // the staged source has been read by every thread
        if (tid == 0) {
          if (o < nout - 1) {
            fence_proxy_async();
            issue(cur, tile, s_sel[o + 1]);
          } else if (nxt.seek(a, tile + gridDim.x)) {
            fence_proxy_async();
            issue(nxt, tile + gridDim.x, s_sel[0]);
          }
        }
      }
      // z factors of this column (kz <= nz/2; pad columns carry zeros anyway),
      // requested before the transform so that their latency is hidden
      const int nz = a.nz;
      const float zf = (ok && kz <= nz / 2) ? __ldg(mult_z + s_zm[o] * nz + kz) : 0.f;
      float zf2 = 0.f;
      if constexpr (DUAL)
        zf2 = (ok && s_dst2[o] != nullptr && kz <= nz / 2) ? __ldg(mult_z + s_zm2[o] * nz + kz) : 0.f;
      if constexpr (kStore) fft_line<N, L, false, V>(v, p, c, s_x, s_tw, wait_store);
      else fft_line<N, L, false, V>(v, p, c, s_x, s_tw);
      const bool mi = s_mi[o] != 0;
      if constexpr (DUAL) {
        float2* d = s_dst[o] + base;
        // outputs with a second store: the same transform with another z
        // factor (displacement components), both stores per register slot so
        // that each slot dies after its two stores
        float2* d2 = s_dst2[o];
        const bool two = ok && d2 != nullptr;
        const bool mi2 = s_mi2[o] != 0;
        d2 = two ? d2 + base : nullptr;
#pragma unroll
        for (int j = 0; j < E; ++j) {
          const size_t off = (size_t)fft_out_index<N, V>(p, j) * nhp;
          float2 w = cscale(v[j], zf);
          if (mi) w = cmuli(w);
          if (ok) d[off] = w;
          if (two) {
            float2 w2 = cscale(v[j], zf2);
            if (mi2) w2 = cmuli(w2);
            d2[off] = w2;
          }
        }
      } else if constexpr (kStore) {
        __syncthreads();  // every thread has read its last exchange values
#pragma unroll
        for (int j = 0; j < E; ++j) {
          float2 w = cscale(v[j], zf);
          if (mi) w = cmuli(w);
          s_x[fft_out_index<N, V>(p, j) * TC + c] = w;
        }
        fence_proxy_async();
        __syncthreads();
        if (tid == 0) {
#pragma unroll
          for (int b = 0; b < GS::kBoxes; ++b)
            tma_store_2d(&a.tm_out[o], kz0, row0 + b * GS::kRows, smem_u32(s_x + b * GS::kRows * TC));
          bulk_commit();
        }
        pending = true;
        continue;
      }
      __syncthreads();
    }
  }
  // columns past the band that the radius before had: zeros
  bool cleared = false;
  for (int g = 0; g < (kMultiRad<N> ? a.rad.n : 1); ++g) {
    if (a.rad.band == nullptr || __ldg(a.rad.wide) != 0) break;
    const int had = a.rad.prev[g] < 0 ? nhp : __ldg(a.rad.band + 4 * a.rad.prev[g] + 2) + 1;
    const int k0 = (__ldg(a.rad.band + 4 * a.rad.ms[g] + 2) + TC) / TC, zt = (had + TC - 1) / TC - k0;
    if (zt <= 0) continue;
    const int nz0 = a.nx * a.batch * zt;
    if constexpr (kStore) {
      if (!cleared) {
        wait_store();
        for (int i = tid; i < N * TC; i += TC * P) s_x[i] = make_float2(0.f, 0.f);
        fence_proxy_async();
        __syncthreads();
        cleared = true;
      }
      if (tid == 0)
        for (int i = blockIdx.x; i < nz0; i += gridDim.x) {
          const int x = i / zt, kz0 = (k0 + i - x * zt) * TC, row0 = (g * 6 * a.nx * a.batch + x) * N;
          for (int o = 0; o < nout; ++o)
#pragma unroll
            for (int b = 0; b < GS::kBoxes; ++b)
              tma_store_2d(&a.tm_out[o], kz0, row0 + b * GS::kRows, smem_u32(s_x + b * GS::kRows * TC));
          bulk_commit();
        }
    } else {
      for (int i = blockIdx.x; i < nz0; i += gridDim.x) {
        const int x = i / zt, kz = (k0 + i - x * zt) * TC + c;
        if (kz >= nhp) continue;
        for (int o = 0; o < nout; ++o)
          for (int r = p; r < N; r += P) {
            const size_t at = ((size_t)x * N + r) * nhp + kz;
            s_dst[o][at] = make_float2(0.f, 0.f);
            if (s_dst2[o] != nullptr) s_dst2[o][at] = make_float2(0.f, 0.f);
          }
      }
    }
  }
  if (kStore && tid == 0) bulk_wait_all();
}

// One x/y tile width: staged tile + exchange + twiddles + multipliers +
// alignment slack, and the block size.
template <int N, int TC, int V = 0> struct CfgXY {
  static constexpr int E = Shape<N, V>::E, P = Shape<N, V>::P, P1 = Shape<N, V>::P1, NTW = Shape<N, V>::kTw;
  static constexpr size_t smem = (size_t)N * TC * 8 + (size_t)XLayoutCols<E, P, TC, P1>::kSize * 8 +
                                 (size_t)NTW * 8 + (size_t)3 * N * 4 + 128;
  static constexpr int threads = TC * P;
};

// The x/y tile widths a plan may run (the autotuner's candidates): the
// default and half of it while a TMA box row stays at least 64 bytes.  Every
// width computes each column's transform with the same arithmetic, so the
// choice changes timings only.
#ifndef PIN_TC_LONG
#define PIN_TC_LONG 16
#endif
// default columns per x/y tile for P threads per line (a TMA box row is TC x 8 bytes)
constexpr int default_tc(int P) { return P >= 16 ? PIN_TC_LONG : (P >= 8 ? 16 : (P == 4 ? 32 : 64)); }
template <int N, int V = 0> struct Tiles {
  static constexpr int T0 = default_tc(Shape<N, V>::P);
  static constexpr int T1 = T0 / 2 >= 8 ? T0 / 2 : T0;
};

template <int N, int TC, int V>
static cudaError_t set_attrs_xy() {
  constexpr int smem = (int)CfgXY<N, TC, V>::smem;
  cudaError_t e = cudaFuncSetAttribute(k_pass_x<N, TC, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_pass_y<N, TC, false, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_pass_y<N, TC, true, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

// both tile widths of one radix schedule
template <int N, int V>
static cudaError_t set_attrs_xy_all() {
  cudaError_t e = set_attrs_xy<N, Tiles<N, V>::T0, V>();
  if (e != cudaSuccess) return e;
  if constexpr (Tiles<N, V>::T1 != Tiles<N, V>::T0) e = set_attrs_xy<N, Tiles<N, V>::T1, V>();
  return e;
}

// Blocks of a kernel resident on the device at once (asked once per kernel and
// process: every device the library runs on is a GB300).
template <auto Kernel>
static long resident(int threads, size_t smem) {
  static const long r = [&] {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, Kernel, threads, smem);
    return (long)std::max(1, sms) * std::max(1, per_sm);
  }();
  return r;
}
// Persistent grid: as many blocks as fit on the device, at most one per tile.
template <auto Kernel>
static unsigned persistent_grid(int threads, size_t smem, long ntiles) {
  return (unsigned)std::min<long>(resident<Kernel>(threads, smem), std::max<long>(1, ntiles));
}

template <int N, int TC, int V>
static cudaError_t run_x(const ArgsX& a_in, cudaStream_t st) {
  using C = CfgXY<N, TC, V>;
  ArgsX a = a_in;
  if (a.rad.n < 1 || (a.rad.n > 1 && !kMultiRad<N>)) return cudaErrorInvalidValue;
  // output maps: the source map's geometry in store boxes, one per output
  for (int f = 0; f < a.nout; ++f) {
    const cudaError_t e = make_tmap_x(&a.tm_out[f], a.dst[f], N, a.ny, a.nhp, a.batch * (3 * a.rad.n - 2), TC,
                                      Store<N>::kBoxes);
    if (e != cudaSuccess) return e;
  }
  const long ntiles = (((long)a.ny * a.nhp + TC - 1) / TC) * a.batch * a.rad.n;
  const unsigned grid = persistent_grid<k_pass_x<N, TC, V>>(C::threads, C::smem, ntiles);
  k_pass_x<N, TC, V><<<grid, C::threads, C::smem, st>>>(a);
  return cudaGetLastError();
}

template <int N, int TC, int V>
static cudaError_t run_y(const ArgsY& a, cudaStream_t st) {
  using C = CfgXY<N, TC, V>;
  const long ntiles = (long)a.nx * a.batch * ((a.nhp + TC - 1) / TC) * a.rad.n;
  bool dual = false;
  for (int o = 0; o < a.nout; ++o) dual = dual || a.dst2[o] != nullptr;
  if (a.rad.n < 1 || (a.rad.n > 1 && (dual || !kMultiRad<N>))) return cudaErrorInvalidValue;
  if (!dual) {
    // output maps: rows (x, ky) of nhp values in store boxes
    ArgsY b = a;
    for (int o = 0; o < b.nout; ++o) {
      const cudaError_t e = make_tmap_rows(&b.tm_out[o], b.dst[o], b.nhp, (long long)b.nx * b.batch * N * (6 * b.rad.n - 5),
                                           TC, Store<N>::kRows);
      if (e != cudaSuccess) return e;
    }
    const unsigned grid = persistent_grid<k_pass_y<N, TC, false, V>>(C::threads, C::smem, ntiles);
    k_pass_y<N, TC, false, V><<<grid, C::threads, C::smem, st>>>(b);
    return cudaGetLastError();
  }
  const unsigned grid = persistent_grid<k_pass_y<N, TC, true, V>>(C::threads, C::smem, ntiles);
  k_pass_y<N, TC, true, V><<<grid, C::threads, C::smem, st>>>(a);
  return cudaGetLastError();
}

// launch with a tile width that is one of Tiles<N, V> (anything else: the default)
template <int N, int V>
static cudaError_t launch_x_v(int tc, const ArgsX& a, cudaStream_t st) {
  return tc == Tiles<N, V>::T1 ? run_x<N, Tiles<N, V>::T1, V>(a, st) : run_x<N, Tiles<N, V>::T0, V>(a, st);
}
template <int N, int V>
static cudaError_t launch_y_v(int tc, const ArgsY& a, cudaStream_t st) {
  return tc == Tiles<N, V>::T1 ? run_y<N, Tiles<N, V>::T1, V>(a, st) : run_y<N, Tiles<N, V>::T0, V>(a, st);
}

template <int N, int V>
static PassShape xy_shape_of() {
  using S = Shape<N, V>;
  constexpr int TC = Tiles<N, V>::T0;
  return PassShape{S::E, S::P, S::P1, S::P2, TC, 0, CfgXY<N, TC, V>::smem, 0, CfgXY<N, TC, V>::threads, 0};
}


}  // namespace pin
