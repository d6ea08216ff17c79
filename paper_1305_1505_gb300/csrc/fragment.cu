// Fragmentation front end (Sec. 2.1.2): the order in which the particles are
// considered (descending F_max; ties by ascending particle index, a reading:
// the paper gives no tie rule) and, per particle, how many of its six grid
// neighbours come before it in that order (0: the particle is a peak of the
// F_max field and starts a new halo, case (i); the sequential accretion and
// merging that follow stay with the caller).
//
// The order is a stable least-significant-digit radix sort of keys that rise as
// F_max falls (F_max >= 0 and never NaN, so its bits order as F does), carrying
// the particle index.  It is bound by memory traffic and by the shared-memory
// reordering, both per pass, so it takes as few passes as the keys need: the
// keys run from 0 (the largest F_max) to umax - umin + 1 (F_max = 0), 26 to 27
// bits on the collapse times of a few radii, three digits of 9 bits; a wider
// range takes a fourth pass (the 40 radii of the benchmark: 28 bits, four of 7).
// One kernel finds the range, one counts every digit of every pass, and each
// pass is a single kernel: a tile's digits are ranked and reordered by digit in
// shared memory, its place among the earlier tiles comes from a look-back over
// their published counts (no histogram pass, scan or table per pass), and runs
// of equal digits go out to consecutive addresses.  Pass 0 reads F_max and
// makes the index on the fly; the last pass writes only the indices.
//
// 768^3, order and counts: 12.2 ms a call in a run of calls, 11.3 for a single
// one, with three passes (4 radii), 14.1 with four (40 radii); 15.8 with a
// histogram pass, a scan of the histogram table and a scatter for each of four
// digits.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "kernels.cuh"

namespace pin {
namespace {

constexpr int kThreads = 512;
constexpr int kItems = 16;
constexpr int kTile = kThreads * kItems;  // keys per block: runs of 16 at 9 bits
constexpr int kWarps = kThreads / 32;
constexpr int kBits = 9;  // at most, per pass
constexpr int kBins = 1 << kBits;
constexpr int kPasses = 4;  // 32 bits at most
static_assert(kBins == kThreads, "one thread per digit");

// The sort of one call, in device memory.
struct Sort {
  unsigned umin, umax;  // smallest non-zero and largest bits of F_max
  int passes, width;    // digits of `width` bits
  unsigned ticket[kPasses];          // tiles started, per pass
  unsigned base[kPasses][kBins];     // counts, then first place, of each digit
};

__device__ __forceinline__ unsigned fkey(float f, unsigned umin, unsigned umax) {
  const unsigned u = __float_as_uint(f);
  return u ? umax - u : umax - umin + 1;
}

__global__ void k_sort_init(Sort* s) {
  for (int i = threadIdx.x; i < kPasses * kBins; i += blockDim.x) s->base[i / kBins][i % kBins] = 0;
  if (threadIdx.x < kPasses) s->ticket[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    s->umin = 0xffffffffu;
    s->umax = 0;
  }
}

// Block-wide range of non-zero bits into the sort's.
__device__ __forceinline__ void add_range(Sort* s, unsigned lo, unsigned hi) {
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if ((threadIdx.x & 31) == 0) {
    if (lo < *(volatile unsigned*)&s->umin) atomicMin(&s->umin, lo);
    if (hi > *(volatile unsigned*)&s->umax) atomicMax(&s->umax, hi);
  }
}

__global__ void __launch_bounds__(256) k_sort_range(const float* __restrict__ fmax, long n, Sort* s) {
  unsigned lo = 0xffffffffu, hi = 0;
  for (long i = blockIdx.x * 256l + threadIdx.x; i < n; i += gridDim.x * 256l) {
    const unsigned u = __float_as_uint(__ldg(fmax + i));
    if (u) lo = min(lo, u);
    hi = max(hi, u);
  }
  add_range(s, lo, hi);
}

// Number of passes and digit width: as few digits of at most kBits as cover
// the largest key.
__global__ void k_sort_plan(Sort* s) {
  if (s->umax == 0) s->umin = 0;  // all zero: one key, 1
  const unsigned top = s->umax - s->umin + 1;
  const int bits = 32 - __clz(top);
  s->passes = (bits + kBits - 1) / kBits;
  s->width = (bits + s->passes - 1) / s->passes;
}

// Digit counts of every pass.
__global__ void __launch_bounds__(512) k_sort_count(const float* __restrict__ fmax, long n, Sort* s) {
  __shared__ unsigned s_h[kPasses][kBins];
  for (int i = threadIdx.x; i < kPasses * kBins; i += 512) s_h[i / kBins][i % kBins] = 0;
  const unsigned umin = s->umin, umax = s->umax;
  const int passes = s->passes, width = s->width;
  const unsigned mask = (1u << width) - 1u;
  __syncthreads();
  constexpr int U = 8;
  const long step = (long)gridDim.x * 512 * U;
  for (long b = (long)blockIdx.x * 512 * U; b < n; b += step) {
    float f[U];
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const long i = b + j * 512 + threadIdx.x;
      f[j] = i < n ? __ldg(fmax + i) : -1.f;
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      if (f[j] < 0.f) continue;
      unsigned k = fkey(f[j], umin, umax);
      for (int p = 0; p < passes; ++p, k >>= width) atomicAdd(&s_h[p][k & mask], 1u);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < passes * kBins; i += 512) {
    const unsigned c = s_h[i / kBins][i % kBins];
    if (c) atomicAdd(&s->base[i / kBins][i % kBins], c);
  }
}

__device__ __forceinline__ unsigned block_exclusive_scan(unsigned v, unsigned* s_warp) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  unsigned x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) s_warp[w] = x;
  __syncthreads();
  if (w == 0) {
    unsigned t = lane < kWarps ? s_warp[lane] : 0u;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, t, d);
      if (lane >= d) t += y;
    }
    if (lane < kWarps) s_warp[lane] = t;  // inclusive warp prefixes
  }
  __syncthreads();
  return (w > 0 ? s_warp[w - 1] : 0u) + x - v;
}

// Counts -> first place of each digit; one block per pass.
__global__ void __launch_bounds__(kThreads) k_sort_base(Sort* s) {
  __shared__ unsigned s_warp[kWarps];
  unsigned* b = s->base[blockIdx.x];
  b[threadIdx.x] = block_exclusive_scan(b[threadIdx.x], s_warp);
}

// Published count of a tile's digit: nothing yet, its own count, or the count
// of it and all earlier tiles.
constexpr unsigned kOwn = 1u << 30, kAll = 2u << 30, kCount = kOwn - 1;  // n3 <= 768^3 < 2^30
// Polls of an earlier tile's count before a block gives up: a poll takes about
// a thousand clocks, so the default is about a second.  The tiles are handed
// out in order by a ticket, so every tile waited for is running or done and
// publishes without waiting for a later one.
constexpr int kPolls = 1 << 21;
constexpr int kPollCycles = 1 << 10;
constexpr int kWindow = 8;
constexpr int kCrowd = 6;  // lanes that lost their slot: 3 to 12 made no difference

// Lanes of the warp that hold the same digit as this one.  The match
// instruction walks the distinct values (57 cycles of its pipe for 32 random
// digits, which bound the passes: 64 % busy, 4.4 ms each on 768^3), and a
// ballot per bit costs more issue slots still.  But few lanes share one of 512
// digits: every lane writes its number to the digit's slot, the lanes that
// find another's there know of a collision, and those groups, about one per
// round, are collected one by one; crowded rounds (the highest digit) fall
// back to the match.
__device__ __forceinline__ unsigned same_digit(unsigned d, int lane, uint8_t* slot) {
  slot[d] = (uint8_t)lane;
  __syncwarp();
  unsigned lost = __ballot_sync(0xffffffffu, slot[d] != lane);
  unsigned peers = 1u << lane;
  if (__popc(lost) > kCrowd) return __match_any_sync(0xffffffffu, d);
  while (lost) {  // the same for all lanes
    const unsigned dl = __shfl_sync(0xffffffffu, d, __ffs(lost) - 1);
    const unsigned with = __ballot_sync(0xffffffffu, d == dl);
    if (d == dl) peers = with;
    lost &= ~with;
  }
  return peers;
}

// One pass.  Warp w owns the tile positions [w * 32 kItems, (w + 1) * 32
// kItems); its lane l holds item i at position w * 32 kItems + 32 i + l, so
// (warp, item, lane) is position order.  Ranks among equal digits are counted
// per warp (lanes holding the same digit in one item round, plus the warp's
// running count of that digit), then offset by the counts of the lower warps.
// The values are loaded while the look-back waits.
__global__ void __launch_bounds__(kThreads, 2) k_sort_pass(const float* __restrict__ fmax, const unsigned* keys_a,
                                                           const unsigned* vals_a, unsigned* keys_b, unsigned* vals_b,
                                                           unsigned* order, int n, int pass, Sort* s,
                                                           unsigned* status, int max_polls, int* err) {
  const int passes = s->passes;
  if (pass >= passes) return;
  extern __shared__ unsigned smem[];
  unsigned* s_k = smem;                                             // [kTile]
  unsigned* s_v = smem + kTile;                                     // [kTile]
  unsigned (*s_cnt)[kBins] = reinterpret_cast<unsigned (*)[kBins]>(smem + 2 * kTile);  // [kWarps][kBins]
  unsigned* s_goff = smem + 2 * kTile + kWarps * kBins;             // [kBins]: first place minus place in the tile
  unsigned* s_start = s_goff + kBins;                               // [kBins]
  uint8_t* s_own = reinterpret_cast<uint8_t*>(s_start + kBins);     // [kWarps][kBins]: same_digit
  __shared__ unsigned s_warp[kWarps], s_tile;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const bool first = pass == 0, last = pass == passes - 1;
  const int width = s->width, shift = pass * width;
  const unsigned mask = (1u << width) - 1u, umin = s->umin, umax = s->umax;
  const unsigned ntiles = (unsigned)((n + kTile - 1) / kTile);
  volatile unsigned* st = status + (size_t)pass * ntiles * kBins + tid;
  unsigned* out = last ? order : vals_b;
  // Nothing to do after a failed wait, whose outputs are incomplete.  Another
  // block may set the word while this one starts, so one thread reads it and
  // the block leaves as a whole: one that lost some of its warps here would
  // rank with counts that were never cleared and write out of range.
  if (__syncthreads_or(tid == 0 && *(volatile int*)err != 0)) return;
  for (;;) {
    if (tid == 0) s_tile = atomicAdd(&s->ticket[pass], 1u);
    for (int j = lane; j < kBins; j += 32) s_cnt[w][j] = 0;
    __syncthreads();
    const unsigned tile = s_tile;
    if (tile >= ntiles) return;
    const int base = (int)(tile * kTile), seg = base + w * 32 * kItems + lane;  // n < 2^30
    const int valid = min(kTile, n - base);
    unsigned key[kItems];
    unsigned short pos[kItems];
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const int idx = seg + 32 * i;
      key[i] = idx >= n ? 0xffffffffu : first ? fkey(__ldg(fmax + idx), umin, umax) : __ldg(keys_a + idx);
    }
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      // positions past the end rank behind all others, in the last digit
      const unsigned d = (key[i] >> shift) & mask;
      const unsigned peers = same_digit(d, lane, s_own + w * kBins);
      const unsigned before = s_cnt[w][d];
      __syncwarp();
      if ((peers & lt) == 0) s_cnt[w][d] = before + __popc(peers);
      __syncwarp();
      pos[i] = (unsigned short)(before + __popc(peers & lt));
    }
    __syncthreads();
    // digit tid: offsets of each warp's run within the digit, and the tile's
    // count, published without the positions past the end
    unsigned acc = 0;
#pragma unroll
    for (int j = 0; j < kWarps; ++j) {
      const unsigned c = s_cnt[j][tid];
      s_cnt[j][tid] = acc;
      acc += c;
    }
    const unsigned own = acc - (tid == (int)mask ? (unsigned)(kTile - valid) : 0u);
    if (ntiles > 1) st[(size_t)tile * kBins] = (tile == 0 ? kAll : kOwn) | own;
    const unsigned start = block_exclusive_scan(acc, s_warp);
    s_start[tid] = start;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const unsigned d = (key[i] >> shift) & mask;
      pos[i] = (unsigned short)(pos[i] + s_start[d] + s_cnt[w][d]);
      s_k[pos[i]] = key[i];
    }
    unsigned (&val)[kItems] = key;  // the keys are in shared memory
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const int idx = seg + 32 * i;
      val[i] = first ? (unsigned)idx : (idx < n ? __ldg(vals_a + idx) : 0u);
    }
    // look back: the counts of the earlier tiles, kWindow of them at a time
    // (all resident blocks start their tiles together, so some 150 tiles back
    // to the last one that knows all its predecessors; one load at a time they
    // took longer than everything else)
    unsigned sum = 0;
    bool gave_up = false;
    int polls = 0;
    for (int t = (int)tile - 1; t >= 0;) {
      unsigned v[kWindow];
#pragma unroll
      for (int k = 0; k < kWindow; ++k) {
        v[k] = kAll;  // before the first tile
        if (t >= k) v[k] = st[(size_t)(t - k) * kBins];
      }
      int seen = 0;
      bool all = false;
#pragma unroll
      for (int k = 0; k < kWindow; ++k) {
        if (all || seen < k || v[k] == 0) continue;
        seen = k + 1;
        sum += v[k] & kCount;
        all = (v[k] & kAll) != 0;
      }
      if (all) break;
      t -= seen;
      if (seen == 0 && ++polls > max_polls) {
        gave_up = true;
        break;
      }
    }
    if (tile > 0 && !gave_up) st[(size_t)tile * kBins] = kAll | (sum + own);
    s_goff[tid] = s->base[pass][tid] + sum - start;
#pragma unroll
    for (int i = 0; i < kItems; ++i) s_v[pos[i]] = val[i];
    if (__syncthreads_or(gave_up)) {
      if (tid == 0) atomicCAS(err, kErrNone, kErrOrder);  // an earlier failure stays the one reported
      return;
    }
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const int q = i * kThreads + tid;
      const unsigned k = s_k[q], place = s_goff[(k >> shift) & mask] + q;
      if (q < valid) {
        if (!last) keys_b[place] = k;
        out[place] = s_v[q];
      }
    }
    __syncthreads();  // the buffers are free for the next tile
  }
}
constexpr size_t kPassSmem = (2 * kTile + kWarps * kBins + 2 * kBins) * sizeof(unsigned) + kWarps * kBins;

// Number of the six periodic neighbours (+-1 along x, y, z) that come before
// particle q in the order: larger F_max, or equal F_max and smaller index.
// Four consecutive z per thread (every nz is a multiple of 8): seven loads for
// four particles in place of 28, which bound it (768^3 1.39 -> 0.80 ms).
__global__ void __launch_bounds__(256) k_neighbours_before(const float* __restrict__ F, int nx, int ny, int nz,
                                                           uint8_t* out) {
  const unsigned n4 = (unsigned)nx * ny * nz / 4, nz4 = nz / 4;
  const float4* F4 = reinterpret_cast<const float4*>(F);
  for (unsigned i = blockIdx.x * 256u + threadIdx.x; i < n4; i += gridDim.x * 256u) {
    const unsigned line = i / nz4;
    const int z4 = (int)(i - line * nz4), x = (int)(line / ny), y = (int)(line - (unsigned)x * ny);
    const int xp = x + 1 == nx ? 0 : x + 1, xm = x == 0 ? nx - 1 : x - 1;
    const int yp = y + 1 == ny ? 0 : y + 1, ym = y == 0 ? ny - 1 : y - 1;
    const unsigned at[4] = {((unsigned)xm * ny + y) * nz4 + z4, ((unsigned)x * ny + ym) * nz4 + z4,
                            ((unsigned)x * ny + yp) * nz4 + z4, ((unsigned)xp * ny + y) * nz4 + z4};
    const unsigned q0 = line * nz;
    const unsigned zl = q0 + (z4 == 0 ? nz - 1 : 4 * z4 - 1), zr = q0 + (4 * z4 + 4 == nz ? 0 : 4 * z4 + 4);
    const float4 f4 = __ldg(F4 + i);
    const float f[6] = {__ldg(F + zl), f4.x, f4.y, f4.z, f4.w, __ldg(F + zr)};
    float g[4][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float4 v = __ldg(F4 + at[k]);
      g[k][0] = v.x;
      g[k][1] = v.y;
      g[k][2] = v.z;
      g[k][3] = v.w;
    }
    const unsigned q = 4 * i;
    unsigned packed = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float c = f[j + 1];
      const unsigned left = j == 0 ? zl : q + j - 1, right = j == 3 ? zr : q + j + 1;
      unsigned n = (f[j] > c) | ((f[j] == c) & (left < q + j));
      n += (f[j + 2] > c) | ((f[j + 2] == c) & (right < q + j));
#pragma unroll
      for (int k = 0; k < 4; ++k) n += (g[k][j] > c) | ((g[k][j] == c) & (at[k] < i));
      packed |= n << (8 * j);
    }
    if (((uintptr_t)out & 3) == 0) {
      reinterpret_cast<unsigned*>(out)[i] = packed;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) out[q + j] = (uint8_t)(packed >> (8 * j));
    }
  }
}

}  // namespace

// Keys and values twice, the published counts of every pass, the sort's words.
static size_t status_bytes(long n3) {
  const long ntiles = (n3 + kTile - 1) / kTile;
  return ntiles > 1 ? (size_t)kPasses * ntiles * kBins * sizeof(unsigned) : 0;  // a single tile looks nowhere
}
size_t fragment_scratch_bytes(long n3) { return (size_t)n3 * 16 + status_bytes(n3) + sizeof(Sort) + 512; }

cudaError_t fragment_order(const float* fmax, int nx, int ny, int nz, void* scratch, int32_t* order,
                           uint8_t* n_before, long long wait_cycles, int* err, cudaStream_t st) {
  const long n3 = (long)nx * ny * nz;
  if (n_before) {
    k_neighbours_before<<<(unsigned)std::min<long>((n3 / 4 + 255) / 256, 152 * 64), 256, 0, st>>>(fmax, nx, ny, nz,
                                                                                                n_before);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (!order) return cudaSuccess;
  unsigned* ka = static_cast<unsigned*>(scratch);
  unsigned *va = ka + n3, *kb = va + n3, *vb = kb + n3;
  unsigned* status = vb + n3;
  Sort* s = reinterpret_cast<Sort*>(((uintptr_t)status + status_bytes(n3) + 255) & ~(uintptr_t)255);
  const unsigned ntiles = (unsigned)((n3 + kTile - 1) / kTile);
  const int max_polls = wait_cycles > 0 ? (int)std::min<long long>(wait_cycles / kPollCycles, kPolls) : kPolls;
  cudaError_t e = cudaFuncSetAttribute(k_sort_pass, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPassSmem);
  if (e == cudaSuccess && ntiles > 1) e = cudaMemsetAsync(status, 0, status_bytes(n3), st);
  if (e != cudaSuccess) return e;
  k_sort_init<<<1, 512, 0, st>>>(s);
  k_sort_range<<<(unsigned)std::min<long>((n3 + 255) / 256, 152 * 8), 256, 0, st>>>(fmax, n3, s);
  k_sort_plan<<<1, 1, 0, st>>>(s);
  k_sort_count<<<(unsigned)std::min<long>((n3 + 4095) / 4096, 152 * 4), 512, 0, st>>>(fmax, n3, s);
  k_sort_base<<<kPasses, kThreads, 0, st>>>(s);
  for (int p = 0; p < kPasses; ++p) {
    const bool odd = p & 1;  // pass 0 writes A, 1 reads A and writes B, ...
    k_sort_pass<<<std::min(ntiles, 2u * 152u), kThreads, kPassSmem, st>>>(fmax, odd ? ka : kb, odd ? va : vb, odd ? kb : ka, odd ? vb : va,
                                                     reinterpret_cast<unsigned*>(order), (int)n3, p, s, status,
                                                     max_polls, err);
  }
  return cudaGetLastError();
}

int fragment_kernels(bool order, bool counts) { return (order ? 5 + kPasses : 0) + (counts ? 1 : 0); }

}  // namespace pin
