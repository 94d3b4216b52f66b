// Shared helpers of libsbr: status/error plumbing, region carving, small vector math.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>

#include "sbr.h"

namespace sbr {

void set_error(const char* fmt, ...);

// Host-side count of kernel launches issued by the library (sbr_launch_count).
void note_launch();

// Streaming multiprocessors of the current device.
int sm_count();

// ---- launches of a chain of dependent kernels ------------------------------
//
// Most calls are chains of kernels of a few microseconds, between which a plain
// launch leaves about 2 us (the previous grid drains, the next is dispatched).  A
// kernel launched by launch_after may be dispatched while the kernel before it in
// the stream still runs; it must not touch global memory before after_previous(),
// which returns once that kernel has finished and its writes are visible.  Every
// thread of such a kernel calls it, so a kernel's end implies the end of all before
// it.  next_may_start(), after the wait, lets the next kernel be dispatched from the
// moment all CTAs of this one have passed it; long kernels leave it out, as waiting CTAs
// hold registers and shared memory that other streams could use.  Called before the wait
// it would let a whole chain in behind one running kernel, and the CTAs that do the work
// next would find the SMs crowded with waiting ones (12 antennas x 128 chirps with
// elevation to points 45.7 us so, 39.1 after the wait; 320 triangles and 4,096 rays to
// points 73.2 and 71.6).  For the same reason a kernel of a few long CTAs, or of many
// small ones sized to fill the chip once, is launched plainly: placed while the kernel
// before still holds some SMs, its CTAs share the others to the end.
//
// What a kernel reads through const __restrict__ pointers or __ldg counts as constant
// for its lifetime, and the compiler may move such a load past a barrier that only
// names memory.  Here it holds from the wait to the kernel's end (the writers have
// finished, and whatever writes next waits for this kernel in turn), so no such load may
// come before the wait.  Hence the loop around it, whose end depends on a value the
// compiler does not know: it moves no load above a branch it cannot decide unless it
// knows the address to be valid, which it does of no pointer argument.  Past the wait
// nothing is stale: the memory operations of all earlier grids are visible to this one,
// and none of its threads has touched their lines before.
template <class T>
struct same_type {
  using type = T;
};
template <class... P>
inline cudaError_t launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                typename same_type<P>::type... args) {
  cudaLaunchConfig_t c{};
  cudaLaunchAttribute a{};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = &a;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, args...);
}
__device__ __forceinline__ void after_previous() {
  unsigned again;  // 0, from the asm the wait is in: the loop is gone from the machine code
  do {
    asm volatile("griddepcontrol.wait;\n\tmov.u32 %0, 0;" : "=r"(again)::"memory");
  } while (again);
}
__device__ __forceinline__ void next_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

constexpr double kC = 299792458.0;  // m/s
constexpr double kTwoPi = 6.283185307179586476925286766559;
constexpr int kAlign = 256;

// Carves sub-regions out of one caller-provided device allocation.  Used twice:
// once with base = nullptr to size the region, once to bind pointers.
struct Carver {
  char* base;
  size_t off = 0;
  explicit Carver(void* b) : base(static_cast<char*>(b)) {}
  template <class T>
  T* take(size_t count) {
    off = (off + kAlign - 1) / kAlign * kAlign;
    T* p = base ? reinterpret_cast<T*>(base + off) : nullptr;
    off += count * sizeof(T);
    return p;
  }
  size_t bytes() const { return (off + kAlign - 1) / kAlign * kAlign; }
};

inline bool aligned256(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 255u) == 0; }

// ---- device scan / sort utilities (scan_sort.cu) --------------------------

// Exclusive scan of n int32 (n from host, or from *d_n when d_n != nullptr with
// n as the capacity).  out[n_actual] receives the total.  scratch needs
// scan_scratch_bytes(capacity).
size_t scan_scratch_bytes(int64_t capacity);
cudaError_t exclusive_scan(const int32_t* in, int32_t* out, int64_t n, const int32_t* d_n,
                           void* scratch, cudaStream_t s);

// Stable LSD radix sort of (key, value) pairs on the low `bits` bits of the
// keys.  Ping-pongs between the two buffers; the sorted result ends in
// keys[0]/vals[0].  n from host, or from *d_n (n = capacity).  Up to
// kSortOneCta keys sort in one CTA with 8-bit digits; d_hist, when not NULL,
// then holds the caller's counts of every digit place (place p's 256 counts at
// [256p, 256p + 256), for the live keys), which spares the CTA its counting
// sweep.  Larger inputs take the multi-CTA path and ignore it.
constexpr int64_t kSortOneCta = 65536;
size_t sort_scratch_bytes(int64_t capacity);
cudaError_t radix_sort_pairs(uint32_t* keys[2], int32_t* vals[2], int64_t n, const int32_t* d_n,
                             int bits, void* scratch, cudaStream_t s, const uint32_t* d_hist = nullptr);

// Lanes of the calling warp (all 32 active) whose 8-bit value d equals this
// lane's, restricted to lanes with ok set: one ballot per bit.
__device__ inline uint32_t warp_peers8(uint32_t d, bool ok) {
  uint32_t m = __ballot_sync(0xffffffffu, ok);
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const uint32_t bit = (d >> b) & 1u;
    const uint32_t bal = __ballot_sync(0xffffffffu, bit);
    m &= bit ? bal : ~bal;
  }
  return m;
}

// ---- order-independent (bitwise deterministic) scatter-add -------------------
//
// Float atomics add in whatever order threads arrive, so such sums change in
// their last bits from run to run.  This scatter adds integers instead, whose sum
// does not depend on the order: pass 1 finds the largest magnitude m among the
// contributions (atomicMax on the float bits), pass 2 adds each contribution x as
// round(x 2^E) to a 64-bit accumulator, E chosen so that 2^log2n contributions of
// magnitude <= m stay below 2^62, and a finishing pass converts acc 2^-E back to
// float.  The resolution 2^-E is about m 2^(log2n - 61), ~1e-12 m for a million
// contributions: far finer than the FP32 sum it replaces.
struct FixScatter {
  unsigned long long* acc;  // zeroed before pass 2
  unsigned int* max_bits;   // zeroed before pass 1
  int log2n;                // ceil(log2(a bound on the number of contributions))
  int alone = 4;            // lanes of a warp with one index that add each for itself (fix_add_peers)
};

__host__ inline int ceil_log2(int64_t n) {
  int l = 0;
  while (l < 62 && ((int64_t)1 << l) < n) ++l;
  return l;
}

// Exponent E for the largest magnitude recorded: m < 2^e with e = biased exponent - 126.
__device__ inline int fix_exp(unsigned int max_bits, int log2n) {
  return 62 - log2n - ((int)((max_bits >> 23) & 0xffu) - 126);
}
// x 2^E rounded to the nearest integer (ties to even) on the integer pipe: the FP64
// pipe, where ldexp and the conversion would run, has a small fraction of its rate.
// Not finite: the values a saturating conversion gives.
__device__ inline long long fix_ll(float x, int E) {
  const unsigned b = __float_as_uint(x), ex = (b >> 23) & 0xffu;
  const long long m = (long long)((b & 0x7fffffu) | (ex ? 0x800000u : 0u));
  const int sh = (int)(ex ? ex : 1u) - 150 + E;
  long long r;
  if (ex == 255u) {
    return x > 0.f ? 0x7fffffffffffffffll : (long long)0x8000000000000000ull;
  } else if (sh >= 0) {
    r = m << min(sh, 39);
  } else if (sh < -25) {
    r = 0;
  } else {
    const long long q = m >> -sh;
    r = (m + ((1ll << (-sh - 1)) - 1) + (q & 1)) >> -sh;
  }
  return (b >> 31) ? -r : r;
}
__device__ inline void fix_add(unsigned long long* acc, float x, int E) {
  atomicAdd(acc, (unsigned long long)fix_ll(x, E));
}

// Sum of x over the lanes of `peers` (all of them call with the same mask): three
// 32-bit warp sums of 26, 26 and 12 bits.
__device__ inline long long peer_sum(unsigned peers, long long x) {
  constexpr unsigned kLow = (1u << 26) - 1u;
  const unsigned lo = __reduce_add_sync(peers, (unsigned)x & kLow);
  const unsigned mid = __reduce_add_sync(peers, (unsigned)(x >> 26) & kLow);
  const int hi = __reduce_add_sync(peers, (int)(x >> 52));
  return (long long)lo + ((long long)mid << 26) + (long long)((unsigned long long)(long long)hi << 52);
}

// Adds the calling lanes' values x[0 .. n) to acc[n i + c], lanes with the same i as
// one: rays of a warp mostly hit the same few triangles, and a large triangle's
// corners take contributions from most of the launch, whose atomics would queue at one
// address.  Integer sums: the result is that of one atomic per lane.  Each group of
// peers runs its warp sums on its own, so groups of up to fs.alone lanes go straight to
// the atomics.
template <int n>
__device__ inline void fix_add_peers(const FixScatter& fs, int i, const float* x, int E) {
  unsigned long long* acc = fs.acc;
  const unsigned peers = __match_any_sync(__activemask(), i);
  if (__popc(peers) <= fs.alone) {
#pragma unroll
    for (int c = 0; c < n; ++c) fix_add(&acc[(size_t)n * i + c], x[c], E);
    return;
  }
  const bool lead = (int)(threadIdx.x & 31) == __ffs(peers) - 1;
#pragma unroll
  for (int c = 0; c < n; ++c) {
    const long long v = peer_sum(peers, fix_ll(x[c], E));
    if (lead) atomicAdd(&acc[(size_t)n * i + c], (unsigned long long)v);
  }
}
__device__ inline float fix_get(unsigned long long a, int E) { return (float)ldexp((double)(long long)a, -E); }
// Warp-reduced max of |x| over the calling warp's lanes (all 32 must call), one atomic per warp.
__device__ inline void fix_note_warp(unsigned int* max_bits, float local_max_abs) {
  const unsigned int b = __reduce_max_sync(0xffffffffu, __float_as_uint(local_max_abs));
  if ((threadIdx.x & 31) == 0 && b) atomicMax(max_bits, b);
}

// Argument validation shared by the entry points (trace.cu).
sbr_status check_radar(const sbr_radar_cfg* r, const char* who);
sbr_status check_grid(const sbr_ray_grid* g, const char* who);

}  // namespace sbr

#define SBR_ARG(cond, ...)                          \
  do {                                              \
    if (!(cond)) {                                  \
      ::sbr::set_error(__VA_ARGS__);                \
      return SBR_ERR_INVALID_ARG;                   \
    }                                               \
  } while (0)

#define SBR_CUDA(call)                                                        \
  do {                                                                        \
    cudaError_t e_ = (call);                                                  \
    if (e_ != cudaSuccess) {                                                  \
      ::sbr::set_error("%s failed: %s", #call, cudaGetErrorString(e_));      \
      return SBR_ERR_CUDA;                                                    \
    }                                                                         \
  } while (0)

// ---- small vector math ------------------------------------------------------

struct d3 {
  double x, y, z;
};
__host__ __device__ inline d3 mk3(double x, double y, double z) { return d3{x, y, z}; }
__host__ __device__ inline d3 operator-(d3 a, d3 b) { return d3{a.x - b.x, a.y - b.y, a.z - b.z}; }
__host__ __device__ inline d3 operator+(d3 a, d3 b) { return d3{a.x + b.x, a.y + b.y, a.z + b.z}; }
__host__ __device__ inline d3 operator*(d3 a, double s) { return d3{a.x * s, a.y * s, a.z * s}; }
__host__ __device__ inline double dot(d3 a, d3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__host__ __device__ inline d3 cross(d3 a, d3 b) {
  return d3{a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}

__host__ __device__ inline float3 f3(float x, float y, float z) { return make_float3(x, y, z); }
__host__ __device__ inline float3 operator-(float3 a, float3 b) { return f3(a.x - b.x, a.y - b.y, a.z - b.z); }
__host__ __device__ inline float3 operator+(float3 a, float3 b) { return f3(a.x + b.x, a.y + b.y, a.z + b.z); }
__host__ __device__ inline float3 operator*(float3 a, float s) { return f3(a.x * s, a.y * s, a.z * s); }
__host__ __device__ inline float dot(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__host__ __device__ inline float3 cross(float3 a, float3 b) {
  return f3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__host__ __device__ inline float l1(float3 a) { return fabsf(a.x) + fabsf(a.y) + fabsf(a.z); }
