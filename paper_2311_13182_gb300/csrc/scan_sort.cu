// Device-wide exclusive scan and stable LSD radix sort (8-bit digits).
//
// Used for path compaction (ray -> first path index), the LBVH's Morton-code
// sort and the point-cloud candidate ordering.  Both are three-phase (tile
// totals, scan of totals, tile-local scan/scatter): no inter-CTA waiting, so no
// kernel here can spin.
#include <stdio.h>

#include <atomic>

#include "cta_sort.cuh"

namespace sbr {
namespace {

constexpr int kThreads = 256;
constexpr int kItems = 8;
constexpr int kTile = kThreads * kItems;

__device__ inline int64_t clamp_n(int64_t cap, const int32_t* d_n) {
  if (!d_n) return cap;
  int64_t n = *d_n;
  return n < 0 ? 0 : (n > cap ? cap : n);
}

// Exclusive scan of one uint32 per thread across the block (blockDim multiple of 32).
// Lanes of packed 16-bit counters scan independently as long as no half overflows.
__device__ inline uint32_t block_exclusive(uint32_t v, uint32_t* total, uint32_t* warp_tot) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[w] = x;
  __syncthreads();
  if (w == 0) {
    uint32_t t = lane < nw ? warp_tot[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    if (lane < nw) warp_tot[lane] = t;
  }
  __syncthreads();
  uint32_t res = (w ? warp_tot[w - 1] : 0u) + x - v;
  *total = warp_tot[nw - 1];
  __syncthreads();
  return res;
}

// A thread's kItems consecutive values (0 beyond n): two 16-byte loads where they are whole and
// aligned (4 M values, sums 7.2 -> 6.0 us, scan 18.6 -> 8.7).
__device__ inline void load_items(const int32_t* in, int64_t base, int64_t n, int32_t (&v)[kItems]) {
  static_assert(kItems == 8, "two int4");
  if (base + kItems <= n && (reinterpret_cast<uintptr_t>(in) & 15) == 0) {
    const int4 a = *reinterpret_cast<const int4*>(in + base), b = *reinterpret_cast<const int4*>(in + base + 4);
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
    return;
  }
#pragma unroll
  for (int i = 0; i < kItems; ++i) v[i] = base + i < n ? in[base + i] : 0;
}

__global__ void k_tile_sums(const int32_t* __restrict__ in, int64_t cap, const int32_t* d_n,
                            int32_t* __restrict__ sums) {
  after_previous();
  next_may_start();
  __shared__ uint32_t wt[32];
  const int64_t n = clamp_n(cap, d_n);
  const int64_t base = (int64_t)blockIdx.x * kTile + (int64_t)threadIdx.x * kItems;
  int32_t v[kItems];
  load_items(in, base, n, v);
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < kItems; ++i) s += (uint32_t)v[i];
  uint32_t tot;
  block_exclusive(s, &tot, wt);
  if (threadIdx.x == 0) sums[blockIdx.x] = (int32_t)tot;
}

// In-place exclusive scan of m values with one CTA (m up to a few million).
__global__ void k_scan_single(int32_t* __restrict__ a, int64_t m) {
  after_previous();
  next_may_start();
  __shared__ uint32_t wt[32];
  uint32_t carry = 0;
  for (int64_t base = 0; base < m; base += blockDim.x) {
    int64_t i = base + threadIdx.x;
    uint32_t v = i < m ? (uint32_t)a[i] : 0u;
    uint32_t tot;
    uint32_t ex = block_exclusive(v, &tot, wt);
    if (i < m) a[i] = (int32_t)(carry + ex);
    carry += tot;
  }
}

__global__ void k_tile_scan(const int32_t* __restrict__ in, int32_t* __restrict__ out, int64_t cap,
                            const int32_t* d_n, const int32_t* __restrict__ sums) {
  after_previous();
  next_may_start();
  __shared__ uint32_t wt[32];
  const int64_t n = clamp_n(cap, d_n);
  if (n == 0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) out[0] = 0;
    return;
  }
  const int64_t base = (int64_t)blockIdx.x * kTile + (int64_t)threadIdx.x * kItems;
  int32_t v[kItems];
  load_items(in, base, n, v);
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < kItems; ++i) s += (uint32_t)v[i];
  uint32_t tot;
  uint32_t run = block_exclusive(s, &tot, wt) + (uint32_t)sums[blockIdx.x];
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const uint32_t x = (uint32_t)v[i];
    v[i] = (int32_t)run;
    run += x;
    if (base + i == n - 1) out[n] = (int32_t)run;
  }
  if (base + kItems <= n && (reinterpret_cast<uintptr_t>(out) & 15) == 0) {
    *reinterpret_cast<int4*>(out + base) = make_int4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<int4*>(out + base + 4) = make_int4(v[4], v[5], v[6], v[7]);
    return;
  }
#pragma unroll
  for (int i = 0; i < kItems; ++i)
    if (base + i < n) out[base + i] = v[i];
}

// ---- radix sort -------------------------------------------------------------

// Three launches per 8-bit digit: the tiles' counts, the scan of each digit's counts over
// the tiles (a CTA per digit), the scatter.  Launches and their latency are what it
// costs up to a few million keys: four passes instead of eight 4-bit ones, 200,000
// pairs 155 -> 63 us of kernels.
constexpr int kDigits = 256;
static_assert(kThreads == kDigits, "a thread per digit");

// Digit of a key at `shift` (mask: the bits sorted by).
__device__ inline uint32_t digit(uint32_t key, int shift, uint32_t mask) { return (key >> shift) & mask; }

// Tile item of (warp, round i, lane): warps hold consecutive runs, rounds within them.
__device__ inline int64_t tile_item(int i) {
  return (int64_t)blockIdx.x * kTile + (threadIdx.x >> 5) * (32 * kItems) + 32 * i + (threadIdx.x & 31);
}

__global__ void __launch_bounds__(kThreads) k_digit_hist(const uint32_t* __restrict__ keys, int64_t cap,
                                                         const int32_t* d_n, int shift, uint32_t mask,
                                                         int32_t* __restrict__ hist, int ntiles) {
  __shared__ uint32_t cnt[kDigits];
  cnt[threadIdx.x] = 0;
  after_previous();
  next_may_start();
  __syncthreads();
  const int64_t n = clamp_n(cap, d_n);
#pragma unroll
  for (int i = 0; i < kItems; ++i) {  // warp-aggregated counts
    const int64_t at = tile_item(i);
    const bool ok = at < n;
    const uint32_t d = ok ? digit(keys[at], shift, mask) : 0u;
    const uint32_t peers = warp_peers8(d, ok);
    if (ok && (int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&cnt[d], (uint32_t)__popc(peers));
  }
  __syncthreads();
  hist[(size_t)threadIdx.x * ntiles + blockIdx.x] = (int32_t)cnt[threadIdx.x];
}

// CTA d: exclusive scan of digit d's counts over the tiles, in place; their sum to total[d].
__global__ void __launch_bounds__(kThreads) k_digit_scan(int32_t* __restrict__ hist, int ntiles,
                                                         int32_t* __restrict__ total) {
  after_previous();
  next_may_start();
  __shared__ uint32_t wt[32];
  int32_t* row = hist + (size_t)blockIdx.x * ntiles;
  uint32_t carry = 0;
  for (int base = 0; base < ntiles; base += kThreads) {
    const int i = base + threadIdx.x;
    const uint32_t v = i < ntiles ? (uint32_t)row[i] : 0u;
    uint32_t sum;
    const uint32_t x = block_exclusive(v, &sum, wt);
    if (i < ntiles) row[i] = (int32_t)(carry + x);
    carry += sum;
  }
  if (threadIdx.x == 0) total[blockIdx.x] = (int32_t)carry;
}

// Stable scatter: a pair's rank among the tile's pairs of its digit is the count of the
// warps before, of the warp's rounds before and of the lanes below; the tile is put in
// order in shared memory first, so that a digit's pairs leave as one run.
__global__ void __launch_bounds__(kThreads) k_digit_scatter(const uint32_t* __restrict__ kin,
                                                            const int32_t* __restrict__ vin,
                                                            uint32_t* __restrict__ kout, int32_t* __restrict__ vout,
                                                            int64_t cap, const int32_t* d_n, int shift, uint32_t mask,
                                                            const int32_t* __restrict__ hist,
                                                            const int32_t* __restrict__ total, int ntiles) {
  __shared__ uint32_t wt[32], cnt[kThreads / 32][kDigits], local[kDigits], skey[kTile];
  __shared__ int32_t sval[kTile], first[kDigits];  // first[d]: output position of the tile's slot 0, for digit d
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < kThreads / 32 * kDigits; i += kThreads) (&cnt[0][0])[i] = 0;
  after_previous();
  next_may_start();
  const int64_t n = clamp_n(cap, d_n);
  uint32_t key[kItems], rank[kItems];
  int32_t val[kItems];
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const int64_t at = tile_item(i);
    key[i] = at < n ? kin[at] : 0u;
    val[i] = at < n ? vin[at] : 0;
  }
  const uint32_t all = (uint32_t)total[threadIdx.x];
  const int32_t before = hist[(size_t)threadIdx.x * ntiles + blockIdx.x];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const bool ok = tile_item(i) < n;
    const uint32_t d = digit(key[i], shift, mask), peers = warp_peers8(d, ok);
    rank[i] = ok ? cnt[w][d] + (uint32_t)__popc(peers & ((1u << lane) - 1u)) : 0u;
    __syncwarp();
    if (ok && lane == __ffs(peers) - 1) cnt[w][d] += (uint32_t)__popc(peers);
    __syncwarp();
  }
  __syncthreads();
  uint32_t sum = 0, unused;
#pragma unroll
  for (int j = 0; j < kThreads / 32; ++j) {  // this thread's digit: exclusive over the warps
    const uint32_t c = cnt[j][threadIdx.x];
    cnt[j][threadIdx.x] = sum;
    sum += c;
  }
  const uint32_t lstart = block_exclusive(sum, &unused, wt), gstart = block_exclusive(all, &unused, wt);
  local[threadIdx.x] = lstart;
  first[threadIdx.x] = (int32_t)(gstart + (uint32_t)before - lstart);
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    if (tile_item(i) >= n) continue;
    const uint32_t d = digit(key[i], shift, mask), at = local[d] + cnt[w][d] + rank[i];
    skey[at] = key[i];
    sval[at] = val[i];
  }
  __syncthreads();
  const int64_t left = n - (int64_t)blockIdx.x * kTile;
  for (int j = threadIdx.x; j < kTile && j < left; j += kThreads) {
    const uint32_t k = skey[j];
    const int32_t at = first[digit(k, shift, mask)] + j;
    kout[at] = k;
    vout[at] = sval[j];
  }
}

inline int tiles_for(int64_t n) { return (int)((n + kTile - 1) / kTile); }

// ---- single-CTA variants for small inputs -----------------------------------
//
// Below kSmall elements a scan runs in one CTA (one launch instead of three),
// and so does a sort of up to kSmall keys: the LBVH's Morton codes (tens of
// thousands of triangles) and the point cloud's detected peaks.

constexpr int kSmall = (int)kSortOneCta;
using cta::kSmallThreads;
using cta::kBitonicMax;
using cta::kSortSmemBytes;

__global__ void __launch_bounds__(kSmallThreads) k_scan_small(const int32_t* __restrict__ in,
                                                              int32_t* __restrict__ out, int64_t cap,
                                                              const int32_t* d_n) {
  after_previous();
  next_may_start();
  __shared__ uint32_t wt[32];
  const int64_t n = clamp_n(cap, d_n);
  uint32_t carry = 0;
  for (int64_t base = 0; base < n; base += (int64_t)kSmallThreads * kItems) {
    const int64_t b = base + (int64_t)threadIdx.x * kItems;
    int32_t v[kItems];
    uint32_t s = 0;
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      v[i] = b + i < n ? in[b + i] : 0;
      s += (uint32_t)v[i];
    }
    uint32_t tot;
    uint32_t run = carry + block_exclusive(s, &tot, wt);
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      if (b + i < n) out[b + i] = (int32_t)run;
      run += (uint32_t)v[i];
    }
    carry += tot;
  }
  if (threadIdx.x == 0) out[n] = (int32_t)carry;
}

__global__ void __launch_bounds__(kSmallThreads) k_sort_small(uint32_t* k0, int32_t* v0, uint32_t* k1,
                                                              int32_t* v1, int64_t cap, const int32_t* d_n,
                                                              int bits, const uint32_t* __restrict__ d_hist) {
  after_previous();
  next_may_start();
  extern __shared__ __align__(16) uint32_t sm[];  // kSortSmemWords
  cta::sort_pairs(k0, v0, k1, v1, clamp_n(cap, d_n), bits, d_hist, sm);
}

// The sort's shared memory exceeds the 48 KB default: raise the limit once per device.
cudaError_t sort_small_attr() {
  static std::atomic<uint64_t> done{0};  // bit per device ordinal below 64
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 64 && ((done.load() >> dev) & 1u)) return cudaSuccess;
  e = cudaFuncSetAttribute(k_sort_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSortSmemBytes);
  if (e == cudaSuccess && dev < 64) done.fetch_or(1ull << dev);
  return e;
}

}  // namespace

size_t scan_scratch_bytes(int64_t capacity) {
  return (size_t)(tiles_for(capacity) + 1) * sizeof(int32_t);
}

cudaError_t exclusive_scan(const int32_t* in, int32_t* out, int64_t n, const int32_t* d_n,
                           void* scratch, cudaStream_t s) {
  if (n <= kSmall) {
    ::sbr::note_launch();
    launch_after(k_scan_small, 1, kSmallThreads, 0, s, in, out, n, d_n);
    return cudaGetLastError();
  }
  const int nt = tiles_for(n < 1 ? 1 : n);
  int32_t* sums = static_cast<int32_t*>(scratch);
  ::sbr::note_launch();
  launch_after(k_tile_sums, nt, kThreads, 0, s, in, n, d_n, sums);
  ::sbr::note_launch();
  launch_after(k_scan_single, 1, 1024, 0, s, sums, nt);
  ::sbr::note_launch();
  launch_after(k_tile_scan, nt, kThreads, 0, s, in, out, n, d_n, sums);
  return cudaGetLastError();
}

size_t sort_scratch_bytes(int64_t capacity) {
  return (size_t)kDigits * (tiles_for(capacity < 1 ? 1 : capacity) + 1) * sizeof(int32_t);
}

cudaError_t radix_sort_pairs(uint32_t* keys[2], int32_t* vals[2], int64_t n, const int32_t* d_n,
                             int bits, void* scratch, cudaStream_t s, const uint32_t* d_hist) {
  if (n <= kSmall) {  // one launch in place of 3 per pass
    cudaError_t e = sort_small_attr();
    if (e != cudaSuccess) return e;
    ::sbr::note_launch();
    launch_after(k_sort_small, 1, kSmallThreads, kSortSmemBytes, s, keys[0], vals[0], keys[1], vals[1], n, d_n, bits,
                 d_hist);
    return cudaGetLastError();
  }
  const int nt = tiles_for(n < 1 ? 1 : n);
  int32_t* hist = static_cast<int32_t*>(scratch);
  int32_t* total = hist + (size_t)kDigits * nt;
  int cur = 0;
  for (int shift = 0; shift < bits; shift += 8) {
    const uint32_t mask = (1u << (bits - shift < 8 ? bits - shift : 8)) - 1u;
    ::sbr::note_launch();
    launch_after(k_digit_hist, nt, kThreads, 0, s, keys[cur], n, d_n, shift, mask, hist, nt);
    ::sbr::note_launch();
    launch_after(k_digit_scan, kDigits, kThreads, 0, s, hist, nt, total);
    ::sbr::note_launch();
    launch_after(k_digit_scatter, nt, kThreads, 0, s, keys[cur], vals[cur], keys[cur ^ 1], vals[cur ^ 1], n, d_n, shift,
                 mask, hist, total, nt);
    cur ^= 1;
  }
  if (cur == 1) {  // odd number of passes: copy back so the result is in buffer 0
    cudaMemcpyAsync(keys[0], keys[1], (size_t)n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s);
    cudaMemcpyAsync(vals[0], vals[1], (size_t)n * sizeof(int32_t), cudaMemcpyDeviceToDevice, s);
  }
  return cudaGetLastError();
}

}  // namespace sbr
