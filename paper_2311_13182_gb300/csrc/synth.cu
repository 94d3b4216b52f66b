// FMCW IF synthesis (Section 3.2.2, Eq. 8) and its adjoint (Eq. 11-12).
//
// cube[v, c, n] = sum_p A_{p,v} exp(j 2 pi (f_c tau_{p,v} + mu tau_{p,v} t_n)),
// t_n = n T / N_s, identical for every chirp c of a static scene.
//
// Split-phase mode (sbr_synthesize's default path): a type-1 non-uniform FFT.  Each
// (path, antenna) is spread onto a periodic grid of 2 N_s points with a width-8
// Kaiser-Bessel kernel, one FFT per antenna follows, and the kernel's Fourier transform
// is divided out: 8 grid updates per (path, antenna) instead of N_s phasors, less than
// 1e-6 from the FP64 sum (details at k_nufft_spread).
//
// Tensor-core kernel (N_s = 256 or 512, run by the allocation-free entry
// point): with n = 16 a + b (b < 16), Eq. 8 factorises per path into
// U_p[a] W_p[b] with U_p[a] = A e^{j 2 pi (phi0 + 16 a delta)} and
// W_p[b] = e^{j 2 pi b delta}, so each antenna's samples are the complex matrix
// product sum_p U_p W_p^T, a GEMM whose contraction runs over the paths.
// Written as a real GEMM with rows (Re, Im) x a, columns b and two contraction
// entries (Re, Im) per path, it goes to mma.sync m16n8k16 with every operand
// split into two fp16 halves (hi + lo, three products hi.hi + hi.lo + lo.hi:
// ~21-bit products) and FP32 accumulation; amplitudes are scaled by a power of
// two per staged chunk so the halves stay in fp16 range (the accumulators are
// rescaled exactly when the scale drops).
//
// Direct FP32 kernel (few records, other sample counts; persistent, one virtual antenna per
// CTA): the CTA's threads own M consecutive samples each and together cover
// all N_s samples, so the sum over paths accumulates in registers with no
// cross-thread reduction.  Paths stream through shared memory in chunks; per
// (path, thread) one split-precision anchor phase (n0 delta_hi is exact in
// FP32, frac() before the low part and phi0 are added) goes through one sincos,
// and the remaining M-1 samples follow by complex rotation with the per-path
// step e^{j 2 pi delta} (4 FP32 multiply/FMA per sample instead of two
// transcendental ops).
//
// Every evaluation writes per-CTA partial sums (or grids) that a second kernel
// adds in a fixed order, so the result is bitwise reproducible.
#include <cooperative_groups.h>
#include <cuda_fp16.h>
#include <limits.h>
#include <math.h>

#include <algorithm>
#include <atomic>
#include <mutex>

#include "common.cuh"
#include "fft.cuh"

namespace sbr {
namespace {

constexpr int kChunk = 512;  // paths staged per chunk (16 KB of shared memory per CTA)
constexpr float kTwoPiF = 6.28318530717958647692f;

// threads per sample group: N_s / 16 (16 samples each), at least 16, at most 256
inline int threads_for(int Ns) {
  int t = Ns / 16;
  return t < 16 ? 16 : (t > 256 ? 256 : t);
}

// Samples after the anchor follow the two-term recurrence of a sampled
// sinusoid, e_{m+1} = 2 cos(w) e_m - e_{m-1} (w = 2 pi delta), one FMA per
// component per sample; its rounding error grows at most linearly in the
// number of steps (|sin(m w) / sin(w)| <= m), so M <= 16 keeps it near 1e-6.
// A CTA has kSplitThreads threads in G = kSplitThreads / (N_s / M) sample
// groups; every group covers all N_s samples and takes every G-th path of each
// staged chunk, and the groups' sums are added through shared memory at the
// end.  (One group per CTA would cap residency at 32 CTAs x 32 threads.)
constexpr int kSplitThreads = 256;

template <int M>
__global__ void __launch_bounds__(kSplitThreads) k_synth_split(const float4* __restrict__ prep, int64_t cap,
                                                               const int32_t* __restrict__ d_P, int V,
                                                               int Q, int Ns, float2* __restrict__ partial) {
  after_previous();
  __shared__ float4 sp[kChunk];
  __shared__ float4 sstep[kChunk];  // cos w, sin w, 2 cos w
  extern __shared__ float2 red[];   // [M][kSplitThreads] when G > 1
  const int T = Ns / M, G = kSplitThreads / T;
  const int g = threadIdx.x / T, lane = threadIdx.x - g * T;
  const int v = blockIdx.x % V, q = blockIdx.x / V;
  const int64_t P = *d_P;
  const int n0 = lane * M;
  const float fn0 = (float)n0;
  // (re, im) pairs advance with packed FP32x2 instructions: one FADD2 per
  // accumulated sample and one FFMA2 per recurrence step
  float2 acc[M];
#pragma unroll
  for (int m = 0; m < M; ++m) acc[m] = make_float2(0.f, 0.f);
  const float4* pv = prep + (size_t)v * cap;
  for (int64_t c0 = (int64_t)q * kChunk; c0 < P; c0 += (int64_t)Q * kChunk) {
    const int cnt = (int)min((int64_t)kChunk, P - c0);
    __syncthreads();
    for (int j = threadIdx.x; j < cnt; j += blockDim.x) {
      const float4 r = pv[c0 + j];
      sp[j] = r;
      float s, c;
      sincospif(2.f * (r.y + r.z), &s, &c);
      sstep[j] = make_float4(c, s, 2.f * c, 0.f);
    }
    __syncthreads();
#pragma unroll 2
    for (int j = g; j < cnt; j += G) {
      const float4 r = sp[j];
      const float4 st = sstep[j];
      float x = fn0 * r.y;  // exact: delta_hi is a multiple of 2^-12 and n0 < 4096
      x -= rintf(x);
      x = fmaf(fn0, r.z, x) + r.x;
      x -= rintf(x);
      float s, c;
      __sincosf(kTwoPiF * x, &s, &c);
      float2 ep = __fmul2_rn(make_float2(r.w, r.w), make_float2(c, s));  // e_0
      acc[0] = __fadd2_rn(acc[0], ep);
      if (M > 1) {
        // e_1 = e_0 e^{jw}
        float2 e = __ffma2_rn(make_float2(-ep.y, ep.y), make_float2(st.y, st.x),
                              __fmul2_rn(make_float2(ep.x, ep.x), make_float2(st.x, st.y)));
        const float2 c2 = make_float2(st.z, st.z);
#pragma unroll
        for (int m = 1; m < M; ++m) {
          acc[m] = __fadd2_rn(acc[m], e);
          if (m + 1 < M) {
            const float2 en = __ffma2_rn(c2, e, make_float2(-ep.x, -ep.y));
            ep = e;
            e = en;
          }
        }
      }
    }
  }
  if (G > 1) {  // add the groups' sums (fixed order: deterministic)
    __syncthreads();
#pragma unroll
    for (int m = 0; m < M; ++m) red[m * kSplitThreads + threadIdx.x] = acc[m];
    __syncthreads();
    if (g != 0) return;
#pragma unroll
    for (int m = 0; m < M; ++m) {
      float2 sum = make_float2(0.f, 0.f);
      for (int gg = 0; gg < G; ++gg) sum = __fadd2_rn(sum, red[m * kSplitThreads + gg * T + lane]);
      acc[m] = sum;
    }
  }
  float2* out = partial + (size_t)blockIdx.x * Ns + n0;
#pragma unroll
  for (int m = 0; m < M; ++m) out[m] = acc[m];
}

// ---- tensor-core forward kernel ---------------------------------------------

// fp16 pair (x0, x1) as hi + lo halves packed in f16x2 registers (lower index low)
__device__ inline void split_h2(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(x0, x1);
  const float2 hf = __half22float2(h);
  const __half2 l = __floats2half2_rn(x0 - hf.x, x1 - hf.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

// c += a b for one m16n8k16 tile (fp16 operands, FP32 accumulators)
__device__ inline void mma_f16(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

constexpr int kMmaThreads = 256;

// MT m16 tiles of a per (Re | Im) block: N_s = 256 MT.  Warp lane (g = lane / 4,
// t = lane % 4) holds, for the 8-path group of one mma k-step, paths 2t and
// 2t + 1 (contraction columns 2t, 2t + 1 for Re and 2t + 8, 2t + 9 for Im),
// rows a = 16 m + g and 16 m + g + 8 of U, and columns b = g, g + 8 of W.
template <int MT>
__global__ void __launch_bounds__(kMmaThreads) k_synth_mma(const float4* __restrict__ prep, int64_t cap,
                                                           const int32_t* __restrict__ d_P, int V, int Q,
                                                           float2* __restrict__ partial) {
  after_previous();
  constexpr int Ns = 256 * MT, NU = 2 * MT;  // U values per (thread, path): a = g + 8 i
  constexpr int kWarps = kMmaThreads / 32;
  // staged records and steps; at the end the warps' sums ([warp][n][Re, Im])
  constexpr int kRed = kWarps * 2 * Ns / 4, kSbuf = kRed > 2 * kChunk ? kRed : 2 * kChunk;
  __shared__ float4 sbuf[kSbuf];
  __shared__ uint32_t wmax[kWarps];
  float4* sp = sbuf;
  float4* sst = sbuf + kChunk;  // e^{j 2 pi 8 delta}, e^{j 2 pi 128 delta}
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int v = blockIdx.x % V, q = blockIdx.x / V;
  const int64_t P = *d_P;
  float acc[2][MT][2][4];  // [Re | Im][m tile][n tile][fragment]
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int d = 0; d < 4; ++d) acc[a][m][c][d] = 0.f;
  int s_run = 126;  // the accumulators hold the sums times 2^s_run
  const float4* pv = prep + (size_t)v * cap;
  const float fa = 16.f * (float)g, fg = (float)g;
  for (int64_t c0 = (int64_t)q * kChunk; c0 < P; c0 += (int64_t)Q * kChunk) {
    const int cnt = (int)min((int64_t)kChunk, P - c0);
    __syncthreads();
    uint32_t m = 0;
    for (int j = threadIdx.x; j < kChunk; j += blockDim.x) {
      const float4 r = j < cnt ? pv[c0 + j] : make_float4(0.f, 0.f, 0.f, 0.f);
      sp[j] = r;
      m = max(m, __float_as_uint(fabsf(r.w)));
      float x8 = 8.f * r.y;  // exact: delta_hi is a multiple of 2^-12
      x8 -= rintf(x8);
      x8 = fmaf(8.f, r.z, x8);
      float x128 = 128.f * r.y;  // exact
      x128 -= rintf(x128);
      x128 = fmaf(128.f, r.z, x128);
      x128 -= rintf(x128);
      float s8, c8, s128, c128;
      __sincosf(kTwoPiF * x8, &s8, &c8);
      __sincosf(kTwoPiF * x128, &s128, &c128);
      sst[j] = make_float4(c8, s8, c128, s128);
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) wmax[warp] = m;
    __syncthreads();
    m = wmax[0];
#pragma unroll
    for (int w = 1; w < kWarps; ++w) m = max(m, wmax[w]);
    if (m == 0u) continue;  // every amplitude of the chunk is zero
    // the chunk's largest |A| lands in [2^14, 2^15): in fp16 range with room for the lo halves
    const int s_c = 14 - ilogbf(__uint_as_float(m));
    if (s_c < s_run) {
      const float f = s_run > 125 ? 1.f : ldexpf(1.f, s_c - s_run);  // exact power of two
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int mm = 0; mm < MT; ++mm)
#pragma unroll
          for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int d = 0; d < 4; ++d) acc[a][mm][c][d] *= f;
      s_run = s_c;
    }
    const float scale = ldexpf(1.f, s_run);
    const int groups = (cnt + 7) >> 3;
    for (int gr = warp; gr < groups; gr += kWarps) {
      float ur[2][NU], ui[2][NU], wr[2][2], wi[2][2];  // [path 2t + h][a index | b = g, g + 8]
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = 8 * gr + 2 * t + h;  // < kChunk; zero records beyond cnt add nothing
        const float4 r = sp[j];
        const float4 st = sst[j];
        float x = fa * r.y;  // exact: 16 g < 128
        x -= rintf(x);
        x = fmaf(fa, r.z, x) + r.x;
        x -= rintf(x);
        float su, cu;
        __sincosf(kTwoPiF * x, &su, &cu);
        const float A = r.w * scale;
        ur[h][0] = A * cu;
        ui[h][0] = A * su;
#pragma unroll
        for (int i = 1; i < NU; ++i) {  // a + 8: n + 128
          ur[h][i] = fmaf(ur[h][i - 1], st.z, -ui[h][i - 1] * st.w);
          ui[h][i] = fmaf(ur[h][i - 1], st.w, ui[h][i - 1] * st.z);
        }
        float y = fg * r.y;  // exact
        y -= rintf(y);
        y = fmaf(fg, r.z, y);
        y -= rintf(y);
        float sw, cw;
        __sincosf(kTwoPiF * y, &sw, &cw);
        wr[h][0] = cw;
        wi[h][0] = sw;
        wr[h][1] = fmaf(cw, st.x, -sw * st.y);  // b + 8
        wi[h][1] = fmaf(cw, st.y, sw * st.x);
      }
      uint32_t Bh[2][2], Bl[2][2];
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        split_h2(wr[0][nt], wr[1][nt], Bh[nt][0], Bl[nt][0]);
        split_h2(wi[0][nt], wi[1][nt], Bh[nt][1], Bl[nt][1]);
      }
      constexpr uint32_t kNeg = 0x80008000u;
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) {
        uint32_t urh[2], url[2], uih[2], uil[2];
        split_h2(ur[0][2 * mt], ur[1][2 * mt], urh[0], url[0]);
        split_h2(ur[0][2 * mt + 1], ur[1][2 * mt + 1], urh[1], url[1]);
        split_h2(ui[0][2 * mt], ui[1][2 * mt], uih[0], uil[0]);
        split_h2(ui[0][2 * mt + 1], ui[1][2 * mt + 1], uih[1], uil[1]);
        // Re rows take (Re U, -Im U) against (Re W, Im W); Im rows take (Im U, Re U)
        const uint32_t Ah_re[4] = {urh[0], urh[1], uih[0] ^ kNeg, uih[1] ^ kNeg};
        const uint32_t Al_re[4] = {url[0], url[1], uil[0] ^ kNeg, uil[1] ^ kNeg};
        const uint32_t Ah_im[4] = {uih[0], uih[1], urh[0], urh[1]};
        const uint32_t Al_im[4] = {uil[0], uil[1], url[0], url[1]};
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
          const uint32_t bh[2] = {Bh[nt][0], Bh[nt][1]}, bl[2] = {Bl[nt][0], Bl[nt][1]};
          mma_f16(acc[0][mt][nt], Ah_re, bh);
          mma_f16(acc[0][mt][nt], Ah_re, bl);
          mma_f16(acc[0][mt][nt], Al_re, bh);
          mma_f16(acc[1][mt][nt], Ah_im, bh);
          mma_f16(acc[1][mt][nt], Ah_im, bl);
          mma_f16(acc[1][mt][nt], Al_im, bh);
        }
      }
    }
  }
  // undo the scale, then add the warps' sums in a fixed order through shared memory
  const float unscale = s_run > 125 ? 0.f : ldexpf(1.f, -s_run);
  __syncthreads();
  float* red = reinterpret_cast<float*>(sbuf);  // [warp][n][Re, Im]
#pragma unroll
  for (int part = 0; part < 2; ++part)
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
      for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int a = 16 * mt + g + ((e & 2) ? 8 : 0);
          const int b = 8 * nt + 2 * t + (e & 1);
          red[warp * 2 * Ns + 2 * (16 * a + b) + part] = acc[part][mt][nt][e] * unscale;
        }
  __syncthreads();
  float2* out = partial + (size_t)blockIdx.x * Ns;
  for (int n = threadIdx.x; n < Ns; n += blockDim.x) {
    float re = 0.f, im = 0.f;
    for (int w = 0; w < kWarps; ++w) {
      re += red[w * 2 * Ns + 2 * n];
      im += red[w * 2 * Ns + 2 * n + 1];
    }
    out[n] = make_float2(re, im);
  }
}

// Per-sample phase in FP64, term by term (the allocation-free entry point):
// x = f_c tau + (B / N_s) tau n, reduced mod 1.
template <int M>
__global__ void __launch_bounds__(256) k_synth_fp64(const float4* __restrict__ prep,
                                                    const float2* __restrict__ plen,
                                                    const float* __restrict__ phase_ofs, int64_t cap,
                                                    const int32_t* __restrict__ d_P, int V, int Q,
                                                    int Ns, double f0, double b_over_ns,
                                                    float2* __restrict__ partial) {
  after_previous();
  __shared__ double2 sx[kChunk];
  __shared__ float sa[kChunk];
  const int v = blockIdx.x % V, q = blockIdx.x / V;
  const int64_t P = *d_P;
  const int n0 = threadIdx.x * M;
  float accr[M], acci[M];
#pragma unroll
  for (int m = 0; m < M; ++m) accr[m] = acci[m] = 0.f;
  for (int64_t c0 = (int64_t)q * kChunk; c0 < P; c0 += (int64_t)Q * kChunk) {
    const int cnt = (int)min((int64_t)kChunk, P - c0);
    __syncthreads();
    for (int j = threadIdx.x; j < cnt; j += blockDim.x) {
      const float2 L = plen[(size_t)v * cap + c0 + j];
      const double t = ((double)L.x + (double)L.y) * (1.0 / kC);
      const double x0 = f0 * t;
      const double d = b_over_ns * t;
      sx[j] = make_double2(x0 - rint(x0) + (double)phase_ofs[c0 + j], d - rint(d));
      sa[j] = prep[(size_t)v * cap + c0 + j].w;
    }
    __syncthreads();
    for (int j = 0; j < cnt; ++j) {
      const double2 xd = sx[j];
      const float a = sa[j];
#pragma unroll
      for (int m = 0; m < M; ++m) {
        double x = fma((double)(n0 + m), xd.y, xd.x);
        x -= rint(x);
        float s, c;
        __sincosf(kTwoPiF * (float)x, &s, &c);
        accr[m] = fmaf(a, c, accr[m]);
        acci[m] = fmaf(a, s, acci[m]);
      }
    }
  }
  float2* out = partial + (size_t)blockIdx.x * Ns + n0;
#pragma unroll
  for (int m = 0; m < M; ++m) out[m] = make_float2(accr[m], acci[m]);
}

// Everything in FP32: tau, f_c tau and mu tau t_n (no split, no FP64).
template <int M>
__global__ void __launch_bounds__(256) k_synth_naive(const float4* __restrict__ prep,
                                                     const float2* __restrict__ plen,
                                                     const float* __restrict__ phase_ofs, int64_t cap,
                                                     const int32_t* __restrict__ d_P, int V, int Q,
                                                     int Ns, float f0, float mu, float dt,
                                                     float2* __restrict__ partial) {
  after_previous();
  __shared__ float2 sx[kChunk];
  __shared__ float so[kChunk];
  const int v = blockIdx.x % V, q = blockIdx.x / V;
  const int64_t P = *d_P;
  const int n0 = threadIdx.x * M;
  float accr[M], acci[M];
#pragma unroll
  for (int m = 0; m < M; ++m) accr[m] = acci[m] = 0.f;
  for (int64_t c0 = (int64_t)q * kChunk; c0 < P; c0 += (int64_t)Q * kChunk) {
    const int cnt = (int)min((int64_t)kChunk, P - c0);
    __syncthreads();
    for (int j = threadIdx.x; j < cnt; j += blockDim.x) {
      sx[j] = make_float2(plen[(size_t)v * cap + c0 + j].x * (float)(1.0 / kC), prep[(size_t)v * cap + c0 + j].w);
      so[j] = phase_ofs[c0 + j];
    }
    __syncthreads();
    for (int j = 0; j < cnt; ++j) {
      const float t = sx[j].x, a = sx[j].y, o = so[j];
#pragma unroll
      for (int m = 0; m < M; ++m) {
        float x = fmaf(mu * t, (float)(n0 + m) * dt, f0 * t) + o;
        x -= rintf(x);
        float s, c;
        __sincosf(kTwoPiF * x, &s, &c);
        accr[m] = fmaf(a, c, accr[m]);
        acci[m] = fmaf(a, s, acci[m]);
      }
    }
  }
  float2* out = partial + (size_t)blockIdx.x * Ns + n0;
#pragma unroll
  for (int m = 0; m < M; ++m) out[m] = make_float2(accr[m], acci[m]);
}

// One thread per (antenna, sample) and group of kRedChirps chirps: the Q per-CTA
// partial sums added in a fixed order (bitwise reproducible), then written to
// the group's chirps (a static scene: every chirp equal).
constexpr int kRedChirps = 16;
__global__ void k_reduce(const float2* __restrict__ partial, int V, int Q, int Ns, int C,
                         float2* __restrict__ cube) {
  after_previous();
  if (C <= kRedChirps) next_may_start();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= V * Ns) return;
  const int v = i / Ns, n = i - v * Ns;
  float re = 0.f, im = 0.f;
  for (int q = 0; q < Q; ++q) {
    const float2 x = partial[((size_t)q * V + v) * Ns + n];
    re += x.x;
    im += x.y;
  }
  const int c1 = min(C, (int)(blockIdx.y + 1) * kRedChirps);
  for (int c = blockIdx.y * kRedChirps; c < c1; ++c) cube[((size_t)v * C + c) * Ns + n] = make_float2(re, im);
}

inline dim3 reduce_grid(int V, int Ns, int C) {
  return dim3((V * Ns + 255) / 256, (C + kRedChirps - 1) / kRedChirps);
}

// ---- adjoint ----------------------------------------------------------------

__global__ void k_chirp_sum(const float2* __restrict__ g, int V, int C, int Ns,
                            float2* __restrict__ gs) {
  after_previous();
  next_may_start();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= V * Ns) return;
  const int v = i / Ns, n = i - v * Ns;
  float re = 0.f, im = 0.f;
  for (int c = 0; c < C; ++c) {
    const float2 x = g[((size_t)v * C + c) * Ns + n];
    re += x.x;
    im += x.y;
  }
  gs[i] = make_float2(re, im);
}

// One thread per (path, antenna): Eq. 12 gives dL/dA = sum_n Re(conj(g_n) e_n),
// Eq. 11 gives dL/dtau = 2 pi A sum_n (f_c + mu t_n) Re(conj(g_n) j e_n); the
// phasor e_n runs by rotation and is re-anchored from the split phase every 32
// samples.  Output per metre of path: dL/dL = dL/dtau / c.
__global__ void __launch_bounds__(256) k_synth_bwd(const float4* __restrict__ prep, int64_t cap,
                                                   const int32_t* __restrict__ d_P, int Ns,
                                                   const float2* __restrict__ gs, float inv_lambda,
                                                   float b_over_cns, float* __restrict__ glen,
                                                   float* __restrict__ gamp, float* __restrict__ gphase) {
  after_previous();
  next_may_start();
  extern __shared__ float2 sg[];
  const int v = blockIdx.y;
  for (int n = threadIdx.x; n < Ns; n += blockDim.x) sg[n] = gs[(size_t)v * Ns + n];
  __syncthreads();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= *d_P) return;
  const float4 r = prep[(size_t)v * cap + p];
  float ss, cs;
  sincospif(2.f * (r.y + r.z), &ss, &cs);
  float sa = 0.f, s0 = 0.f, s1 = 0.f;
  for (int nb = 0; nb < Ns; nb += 32) {
    const float fn = (float)nb;
    float x = fn * r.y;
    x -= rintf(x);
    x = fmaf(fn, r.z, x) + r.x;
    x -= rintf(x);
    float s, c;
    __sincosf(kTwoPiF * x, &s, &c);
    float t0 = 0.f, t1 = 0.f;
#pragma unroll 8
    for (int m = 0; m < 32; ++m) {
      const float2 g = sg[nb + m];
      sa = fmaf(g.x, c, fmaf(g.y, s, sa));
      const float im = fmaf(g.y, c, -g.x * s);
      t0 += im;
      t1 = fmaf((float)m, im, t1);
      const float nc = fmaf(c, cs, -s * ss);
      const float ns = fmaf(c, ss, s * cs);
      c = nc;
      s = ns;
    }
    s0 += t0;
    s1 += fmaf(fn, t0, t1);
  }
  gamp[(size_t)v * cap + p] = sa;
  glen[(size_t)v * cap + p] = kTwoPiF * r.w * fmaf(inv_lambda, s0, b_over_cns * s1);
  // a phase offset o (cycles) enters every sample as e^{j 2 pi o}: dL/do = 2 pi A sum_n Re(conj(g_n) j e_n)
  if (gphase) gphase[(size_t)v * cap + p] = kTwoPiF * r.w * s0;
}

// ---- non-uniform FFT forward kernel -----------------------------------------
//
// The samples are computed as a type-1 non-uniform FFT (Dutt & Rokhlin 1993;
// Kaiser-Bessel kernel, Greengard & Lee 2004, Barnett et al. 2019) instead of
// term by term.  With n = n' + N_s / 2 (n' in [-N_s/2, N_s/2)),
//   S[n] = sum_p c_p e^{j 2 pi n' delta_p},  c_p = A_p e^{j 2 pi (phi0_p + (N_s/2) delta_p)},
// every path is spread onto a periodic grid of M = 2 N_s points, u_p = M delta_p,
//   b[l] = sum_p c_p psi(l - u_p),  psi(x) = I0(beta sqrt(1 - (2x/w)^2)) / I0(beta), |x| < w/2,
// then B[k] = sum_l b[l] e^{+j 2 pi k l / M} (one M-point FFT) and, by Poisson
// summation, S[n' + N_s/2] = B[n'] / Psi(n'/M) with Psi the Fourier transform of
// psi, up to the aliasing terms Psi(n'/M - k), k != 0 (7e-8 relative rms over
// the band for w = 8, beta = 2.3 w at upsampling 2).  Per (path, antenna) that
// is w = 8 kernel values instead of N_s phasors.
//
// The grid position keeps the split phase's precision: M delta_hi is exact in
// FP32 (delta_hi is a multiple of 2^-12, M <= 8192), so the offset t of the path
// from its grid cell carries about 2^-24 of one grid step.  With t = s + 1/2 the
// eight values psi((j - 7/2) - s) are polynomials of degree 8 in s (1.2e-8 of the
// peak), mirrored in pairs, psi_j(s) = E_j(s^2) + s O_j(s^2) = psi_{7-j}(-s): 37
// FMAs for the eight, and no square root or exponential.
//
// One lane takes one record, and its sixteen additions go to the CTA's grid in
// shared memory as integer atomics: the sums are then exact, do not depend on
// the order, and are bitwise reproducible.  A grid word has kNuCopies copies,
// one per lane pair (l, l + 16), and the lower half of a warp adds real parts
// while the upper adds imaginary parts (then the other way round), so the 32
// lanes of an atomic always hit 32 different banks, whatever the cells are:
// neighbouring rays share cells, and consecutive records jump between a ray's
// bounces.  A term is rounded to 2^-25 to 2^-24 of the largest amplitude of its class
// (nu_class: nearly always its chunk of 1,024 records), so that a chunk's additions to
// one copy stay below 2^31; after each class the copies of the touched cells (a flag
// per eight cells) are summed, scaled and added to the CTA's FP32 grid, each point by
// one thread.  The CTAs' grids are added in a fixed order by the finishing kernel.
//
// A CTA has a barrier for a chunk's largest amplitude and one before its sums are added
// up; the next chunk's records are in flight meanwhile, and its preparation needs none.
// Bound by issue slots (209 instructions per 32 records) and the conversion unit,
// three CTAs per SM: 12 antennas x 367,500 records x 256 samples 35 us (109 us when
// each warp kept runs of equal cells in registers, eight lanes to a record, and
// flushed them to its own FP32 grid, one group at a time; 93 us with the chunk sorted
// by cell first), 71 MB of records at 2 TB/s.  A block of 512 cells, so that long
// chirps keep three CTAs per SM too: 4 antennas x 3.1 M records x 4096 samples 250 ->
// 124 us against a block of 1024 in one CTA of 1024 threads.  Error against FP64 over
// the same records 2e-7 (1.3e-6 with the former kernel's approximate sine, square root
// and exponential).
constexpr int kNuW = 8;        // kernel width in grid points
constexpr int kNuCopies = 16;  // copies of a grid word
constexpr int kNuBlock = 512;  // cells a CTA's grid holds at once (71 KB: three CTAs per SM); larger grids block by block
constexpr int kNuThreads = 256;
constexpr int kNuItems = 4;    // records per thread and chunk
constexpr int kNuChunk = kNuThreads * kNuItems;
constexpr int kNuBits = 25;    // 2 kNuChunk / 32 additions per copy of terms up to 0.98 2^25: below 2^31
static_assert(kNuChunk / kNuCopies <= 1 << (31 - kNuBits), "a class's additions to one copy");
constexpr int kNuSpan = 24;    // mean distance of a class's amplitudes from its largest, in eighths of an octave
constexpr int kNuFar = 40;     // the same where their rms is near it all the same
constexpr double kNuBeta = 2.3 * kNuW;

struct NufftCoef {
  // psi((j - 7/2) - s) = sum_k e[k][j] s^(2k) + s sum_k o[k][j] s^(2k), j < 4, |s| <= 1/2
  float e[5][4], o[4][4];
  float inv[9];  // 1 / Psi(n'/M) = sum_k inv[k] (2 n' / N_s)^(2k)
};

// What a record's rate turns into over the chirps, as FP32 pairs: carrier cycles and
// delta per (m/s) of dL/dt.  A product with a rate keeps the fraction of its cycles to
// 2^-25 however many they are; rounded with its whole cycles it would lose a bit for each
// doubling, and a tile's turns would add that up (the last of 16 chirps at up to 100 m/s:
// 2.3e-6 from FP64, 7e-7 so; of 128 chirps at up to 8 m/s 1.7e-6 and 4e-7).
struct Pair32 {
  float hi, lo;
  Pair32() = default;
  __host__ __device__ explicit Pair32(double x) : hi((float)x), lo((float)(x - (double)(float)x)) {}
  // r x - p, p = r hi rounded
  __device__ __forceinline__ float rest(float r, float p) const { return fmaf(r, lo, fmaf(r, hi, -p)); }
};

struct NufftArg {
  int log_m;
  float half_n, m;           // N_s / 2, M = 2 N_s
  double cyc, cell;          // FP64 phase: carrier cycles at n' = 0 and grid cells per metre of path
  double f0_c, b_cn;         // f_c / c and B / (c N_s) per metre
  int V, Q, chirps, chirp0;  // antennas, CTAs per antenna and chirp, chirps of this launch, the first of them
  double per_chirp;          // moving scenes: change of path length per chirp per (m/s) of dL/dt
  // a tile of chirps, per (m/s): the first chirp's carrier cycles and delta, a chirp's turn at n' = 0 and move in cells
  Pair32 cyc0, eps0, turn;
  float move;
};

// Cells a CTA's grid holds, and its points: the cells and w - 1 more to the right
// (folded back, or into the neighbouring block, when the chunk is added up).
__host__ __device__ constexpr int nu_cells(int M) { return M < kNuBlock ? M : kNuBlock; }
__host__ __device__ constexpr int nu_points(int M) { return nu_cells(M) + kNuW; }

// The eight weights psi((j - 7/2) - s): left[j] of point j and right[j] of point 7 - j,
// j < 4, two points per packed FMA.
__device__ __forceinline__ void nu_weights(const NufftCoef& co, float s, float (&left)[4], float (&right)[4]) {
  const float2 s2 = make_float2(s * s, s * s), ss = make_float2(s, s);
#pragma unroll
  for (int j = 0; j < 4; j += 2) {
    float2 E = make_float2(co.e[4][j], co.e[4][j + 1]), O = make_float2(co.o[3][j], co.o[3][j + 1]);
#pragma unroll
    for (int k = 3; k >= 0; --k) E = __ffma2_rn(E, s2, make_float2(co.e[k][j], co.e[k][j + 1]));
#pragma unroll
    for (int k = 2; k >= 0; --k) O = __ffma2_rn(O, s2, make_float2(co.o[k][j], co.o[k][j + 1]));
    O = __fmul2_rn(O, ss);
    left[j] = E.x + O.x;
    left[j + 1] = E.y + O.y;
    right[j] = E.x - O.x;
    right[j + 1] = E.y - O.y;
  }
}

// I0(2 sqrt(q)) by its power series (the terms are positive: no cancellation; q < 100).
constexpr double bessel_i0_of(double q) {
  double t = 1.0, s = 1.0;
  for (int k = 1; k < 200 && t > 1e-18 * s; ++k) {
    t *= q / ((double)k * k);
    s += t;
  }
  return s;
}

// c w rounded to an integer.  Below 2^22 (the outer points: psi <= psi(2) = 0.0914 from
// two grid steps on, terms up to 3.0e6) by one FMA against 1.5 2^23 and the bits'
// difference, which leaves the conversion unit, a quarter of the FMA pipe's rate, to the
// inner points.
constexpr int kNuSmall = 2;  // outer points on either side
constexpr double nu_outer(double x) {  // psi(x)
  return bessel_i0_of(0.25 * kNuBeta * kNuBeta * (1.0 - (2.0 * x / kNuW) * (2.0 * x / kNuW))) /
         bessel_i0_of(0.25 * kNuBeta * kNuBeta);
}
static_assert(0.98 * (1 << kNuBits) * nu_outer(kNuW / 2 - kNuSmall) < 0.99 * (1 << 22),
              "outer terms pass the FMA's range");
__device__ __forceinline__ int nu_term(float c, float w, bool small) {
  return small ? __float_as_int(fmaf(c, w, 12582912.f)) - 0x4B400000 : __float2int_rn(c * w);
}

// An amplitude's logarithm in eighths of an octave (2047 and 2046: not finite).
__device__ __forceinline__ int nu_log(float a) { return (int)((__float_as_uint(a) & 0x7fffffffu) >> 20); }

// The class of records that one pass rounds on one scale, 2^s for the largest amplitude
// (its bits: top) to land in (0.49, 0.98] 2^kNuBits: all N that are left if their
// logarithms (sum: logs) lie within kNuSpan of the largest's on average, or within
// kNuFar with a rms amplitude of an eighth of it or more (nu_one_class); else those within
// kNuSpan of it.  The class's rms amplitude is then an eighth of its largest or more, and
// the rounding stays near the error of the transform around it; on one scale for all, a
// chunk's few strong records would cost its weak ones their bits (one record in 1,024 a
// hundred times the others: 9e-7 to 1.4e-6 from FP64 instead of 1.8e-7; two in 1,024 a
// thousand times the others and cancelling: 3e-5 instead of 1.9e-7).  The returns of one
// chunk differ little: the traced paths of 28 scenes leave kNuSpan in up to 9 % of their
// chunks (two of them in 26 and 39 %), and need a second class in up to 0.1 % (1 %).
// The scale is a power of two, exact; one past a float's range (amplitudes
// below 1e-31) is applied in two factors.
// With the words per chunk that this takes, and the copies added up without sign
// extensions, 12 antennas x 367,500 records went from 41.7 to 40.4 us for the whole
// synthesis, 4 antennas x 3.1 M records x 4096 samples from 122.0 to 123.4, moving chirps
// from 3.50 to 3.31 ms.
struct NuClass {
  float up, down;    // 2^s and its reciprocal
  float more, less;  // the scale's second factor and its reciprocal
  int floor;         // logarithms from here on belong to the class; 0: every record left
  bool rare;         // the fields above are nu_rare's to set
};
__device__ __forceinline__ NuClass nu_class(uint32_t top, int logs, int N) {
  NuClass c;
  const int e = (int)((top + 0x51eb9u) >> 23);  // the largest's exponent, one more from 1.96 2^e on
  c.up = __int_as_float((127 + 126 + kNuBits - e) << 23);
  c.down = __int_as_float((e + 1 - kNuBits) << 23);
  c.more = c.less = 1.f;
  c.floor = 0;
  c.rare = N * ((int)(top >> 20) - kNuSpan) > logs || e < kNuBits;
  return c;
}
__device__ __forceinline__ void nu_rare(NuClass& c, uint32_t top, int logs, int N) {
  const int e = (int)((top + 0x51eb9u) >> 23), l = (int)(top >> 20) - kNuSpan;
  if (e < kNuBits) {  // up would pass a float's range, down fall below it
    c.up = __int_as_float((127 + 126) << 23);
    c.down = __int_as_float((127 - 126) << 23);
    c.more = __int_as_float((127 + kNuBits - e) << 23);
    c.less = __int_as_float((127 - kNuBits + e) << 23);
  }
  c.floor = N * l > logs ? max(l, 0) : 0;
}

// Amplitude whose square counts for nu_one_class: the largest's is 15,000 to 63,000.
__device__ __forceinline__ float nu_part(float a, const NuClass& c) { return a * c.more * c.up * 0x1p-17f; }
__device__ __forceinline__ bool nu_one_class(const NuClass& c, uint32_t top, int power, int logs, int N) {
  const float x = nu_part(__uint_as_float(top), c);
  return power >= (N * (int)(x * x)) >> 6 && N * (c.floor + kNuSpan - kNuFar) <= logs;
}

// Grid words in shared memory are kept kNuZero off, so that the copies add up unsigned,
// with carries and no sign extension.
constexpr uint32_t kNuZero = 0x80000000u;
__device__ __forceinline__ uint4 nu_zero() { return make_uint4(kNuZero, kNuZero, kNuZero, kNuZero); }

// The copies of a grid word (at uint4 index w0; the four 16-byte words in an order that
// gives the lanes of a shared-memory phase different banks) summed and zeroed.
__device__ __forceinline__ long long nu_add_up(uint4* g, int w0, int turn) {
  unsigned long long t = 0;
#pragma unroll
  for (int k = 0; k < kNuCopies / 4; ++k) {
    const int w = w0 + ((k + turn) & (kNuCopies / 4 - 1));
    const uint4 x = g[w];
    g[w] = nu_zero();
    t += (unsigned long long)x.x + x.y + x.z + x.w;
  }
  return (long long)(t - (unsigned long long)kNuCopies * kNuZero);
}

// x = rint(x) + the returned fraction in [-1/2, 1/2], |x| < 2^50; n gets rint(x) mod 2^32.
__device__ __forceinline__ double split_rint(double x, int& n) {
  const double k = x + 6755399441055744.0;  // 1.5 2^52: the integer in the low word
  n = __double2loint(k);
  return x - (k - 6755399441055744.0);
}

// r x modulo 1
__device__ __forceinline__ float cycles_of(float r, const Pair32& x) {
  const float p = r * x.hi;
  return (p - rintf(p)) + x.rest(r, p);
}
// The record's phi0 and delta after a shift of r cyc and r eps; whole multiples of 2^-12
// of the delta shift move into delta_hi (which stays exact).
__device__ __forceinline__ void shift_record(float4& rec, float r, const Pair32& cyc, const Pair32& eps) {
  const float ph = rec.x + cycles_of(r, cyc);
  rec.x = ph - rintf(ph);
  const float p = r * eps.hi, kq = rintf((p + rec.z) * 4096.f), dh = rec.y + kq * (1.f / 4096.f);
  rec.y = dh - rintf(dh);
  rec.z = (p - kq * (1.f / 4096.f)) + (rec.z + eps.rest(r, p));
}

// CTA (q, v, chirp) spreads its share of antenna v's records, P/Q consecutive
// ones.  Writes the CTA's grid, grids[CTA][l].  kBlocks: M > kNuBlock.
template <bool kFp64, bool kMoving, bool kBlocks>
__global__ void __launch_bounds__(kNuThreads, 3)
    k_nufft_spread(const float4* __restrict__ prep, const float2* __restrict__ plen, const float* __restrict__ phase_ofs,
                   const float* __restrict__ rate, int64_t cap, const int32_t* __restrict__ d_P, const NufftArg na,
                   const __grid_constant__ NufftCoef co, float2* __restrict__ grids, unsigned int* __restrict__ fin_cnt) {
  extern __shared__ uint4 nsm[];
  __shared__ uint32_t s_max[2], s_blk[2];     // by the parity of the chunk: largest amplitude, blocks
  __shared__ int s_log[2], s_pow[2];          // and the sums of the amplitudes' logarithms and, rarely, powers
  __shared__ int flag[2][kNuBlock / 8];       // by the parity of the pass: a record of cells 8 o .. 8 o + 7
  const int M = 1 << na.log_m, bs = nu_cells(M), npts = nu_points(M);
  int* grid = reinterpret_cast<int*>(nsm);                            // [npts][re, im][kNuCopies]
  float* sum = reinterpret_cast<float*>(grid + npts * 2 * kNuCopies); // [npts][re, im]: finished chunks
  const int tid = threadIdx.x, lane = tid & 31;
  const int cl = blockIdx.x % na.chirps, v = (blockIdx.x / na.chirps) % na.V, q = blockIdx.x / (na.chirps * na.V);
  const double dt = kMoving ? (double)(na.chirp0 + cl) * na.per_chirp : 0.0;  // path length change per (m/s)
  const Pair32 cyc(dt * na.f0_c), eps(dt * na.b_cn);
  float2* out = grids + (size_t)blockIdx.x * M;
  for (int i = tid; i < npts * (2 * kNuCopies / 4); i += kNuThreads) nsm[i] = nu_zero();
  for (int i = tid; i < 2 * npts; i += kNuThreads) sum[i] = 0.f;
  for (int i = tid; i < 2 * (kNuBlock / 8); i += kNuThreads) (&flag[0][0])[i] = 0;
  if (tid < 2) s_max[tid] = s_blk[tid] = 0u, s_log[tid] = s_pow[tid] = 0;
  after_previous();
  if (blockIdx.x == 0)
    for (int i = tid; i < na.V * na.chirps; i += kNuThreads) fin_cnt[i] = 0u;  // the finishing kernel's counters
  if (kBlocks)
    for (int i = tid; i < M; i += kNuThreads) out[i] = make_float2(0.f, 0.f);
  const int64_t P = *d_P;
  const int64_t r0 = P * q / na.Q;
  const int n = (int)(P * (q + 1) / na.Q - r0);
  const size_t at = (size_t)v * cap + r0;
  const float4* pv = prep + at;
  const bool upper = lane >= 16;
  int* mine = grid + (lane & 15);
  int blk = 0;       // block of cells the grid holds
  int pass = 0;      // passes so far (a chunk has one per block of cells it touches)
  bool bad = false;  // a record that is not finite: the antenna's samples are NaN
  // the finished sums of block blk into the CTA's output (several blocks only)
  auto store_block = [&]() {
    for (int i = tid; i < npts; i += kNuThreads) {
      float2* o = out + ((blk * bs + i - (kNuW / 2 - 1)) & (M - 1));
      *o = make_float2(o->x + sum[2 * i], o->y + sum[2 * i + 1]);
      sum[2 * i] = sum[2 * i + 1] = 0.f;
    }
  };
  float4 rec[kNuItems];  // a chunk's records; then cos, sin of the carrier phase at n' = 0, s, A
  auto load = [&](int c0) {
#pragma unroll
    for (int u = 0; u < kNuItems; ++u) {
      const int p = c0 + tid + u * kNuThreads;
      rec[u] = p < n ? __ldg(&pv[p]) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  load(0);
  __syncthreads();
  // A turn takes a class of a chunk's records: nearly always all of them.  (The votes below
  // are over equal conditions: what depends on a vote stays out of the lanes' registers and
  // needs no reconvergence, 124.6 against 127.2 us for 4 x 3.1 M records x 4096 samples.)
  bool again = false;                     // the turn has another class of the same chunk
  int ceil = 0, left = min(kNuChunk, n);  // logarithms done, records to do of that chunk
  for (int c0 = 0, chunk = 0; c0 < n; ++chunk) {
    int cell[kNuItems], logs = 0;
    uint32_t am = 0, blocks = 0;
#pragma unroll
    for (int u = 0; u < kNuItems; ++u) {
      const int p = c0 + tid + u * kNuThreads;
      float4 r = rec[u];
      float x, t;
      int ce;
      if (kFp64) {
        float2 L2 = make_float2(0.f, 0.f);
        float po = 0.f, ld = 0.f;
        if (p < n) {
          L2 = __ldg(&plen[at + p]);
          po = __ldg(&phase_ofs[r0 + p]);
          if (kMoving) ld = __ldg(&rate[at + p]);
        }
        double L = (double)L2.x + (double)L2.y;
        if (kMoving) L = fma(dt, (double)ld, L);
        int whole;
        x = (float)split_rint(na.cyc * L, whole) + po;
        t = (float)split_rint(fma(na.cell, L, -0.5), ce);  // the cell is rint(u - 1/2), s the rest
        bad |= !isfinite(x + t + r.w);
      } else {
        if (kMoving) {
          const float ld = p < n ? __ldg(&rate[at + p]) : 0.f;
          shift_record(r, ld, cyc, eps);
        }
        x = na.half_n * r.y;  // exact
        x -= rintf(x);
        x = fmaf(na.half_n, r.z, x) + r.x;
        const float uh = na.m * r.y;  // exact
        float fl = floorf(uh);
        t = fmaf(na.m, r.z, uh - fl);
        ce = (int)fl;
        bad |= !isfinite(x + t + r.w);
        fl = floorf(t);
        t = (t - fl) - 0.5f;
        ce += (int)fl;
      }
      ce &= M - 1;
      float sn, cs;
      sincospif(2.f * x, &sn, &cs);
      rec[u] = make_float4(cs, sn, t, r.w);
      cell[u] = ce;
      if (kBlocks && p < n) blocks |= 1u << (ce / kNuBlock);
    }
    if (again) {
#pragma unroll
      for (int u = 0; u < kNuItems; ++u)
        if (nu_log(rec[u].w) >= ceil) rec[u].w = 0.f;
    }
#pragma unroll
    for (int u = 0; u < kNuItems; ++u) {
      am = max(am, __float_as_uint(fabsf(rec[u].w)));
      logs += nu_log(rec[u].w);
    }
    am = __reduce_max_sync(0xffffffffu, am);
    logs = __reduce_add_sync(0xffffffffu, logs);
    if (kBlocks) blocks = __reduce_or_sync(0xffffffffu, blocks);
    if (lane == 0) {
      atomicMax(&s_max[chunk & 1], am);
      atomicAdd(&s_log[chunk & 1], logs);
      if (kBlocks) atomicOr(&s_blk[chunk & 1], blocks);
    }
    __syncthreads();  // the chunk's words; the turn before is added up
    logs = s_log[chunk & 1];
    const uint32_t top = s_max[chunk & 1];
    NuClass cls = nu_class(top, logs, left);
    blocks = kBlocks ? __reduce_or_sync(0xffffffffu, s_blk[chunk & 1]) : 1u;
    again = false;
    if (__any_sync(0xffffffffu, cls.rare)) {  // the same for the whole CTA
      nu_rare(cls, top, logs, left);
      if (cls.floor) {
        float x = 0.f;
#pragma unroll
        for (int u = 0; u < kNuItems; ++u) {
          const float y = nu_part(rec[u].w, cls);
          x = fmaf(y, y, x);
        }
        const int power = __reduce_add_sync(0xffffffffu, (int)x);
        if (lane == 0) atomicAdd(&s_pow[chunk & 1], power);
        __syncthreads();
        if (nu_one_class(cls, top, s_pow[chunk & 1], logs, left)) cls.floor = 0;
      }
      again = __any_sync(0xffffffffu, cls.floor != 0);
      ceil = cls.floor;
      if (again || cls.more != 1.f) {
#pragma unroll
        for (int u = 0; u < kNuItems; ++u) {
          const bool in = nu_log(rec[u].w) >= cls.floor;
          if (again) left -= __syncthreads_count(in);
          rec[u].w = in ? rec[u].w * cls.more : 0.f;
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kNuItems; ++u) rec[u].w *= cls.up;
    c0 += again ? 0 : kNuChunk;
    left = again ? left : min(kNuChunk, n - c0);
    // the turn before's words: read before this turn's first barrier
    if (tid == 0) s_max[~chunk & 1] = s_blk[~chunk & 1] = 0u, s_log[~chunk & 1] = s_pow[~chunk & 1] = 0;
    while (blocks) {
      const int b = kBlocks ? __ffs(blocks) - 1 : 0;
      blocks &= blocks - 1;
      if (kBlocks && b != blk) {  // the same for the whole CTA
        store_block();
        blk = b;
        __syncthreads();
      }
      int* fl = flag[pass & 1];
      if (tid < kNuBlock / 8) flag[~pass & 1][tid] = 0;  // read before this pass
#pragma unroll
      for (int u = 0; u < kNuItems; ++u) {
        const int idx = kBlocks ? cell[u] - b * bs : cell[u];
        if ((kBlocks && (unsigned)idx >= (unsigned)bs) || rec[u].w == 0.f) continue;
        const float a = rec[u].w;
        const float c1 = a * (upper ? rec[u].y : rec[u].x), c2 = a * (upper ? rec[u].x : rec[u].y);
        int* g1 = mine + idx * (2 * kNuCopies) + (upper ? kNuCopies : 0);
        int* g2 = mine + idx * (2 * kNuCopies) + (upper ? 0 : kNuCopies);
        fl[idx >> 3] = 1;
        float wl[4], wr[4];
        nu_weights(co, rec[u].z, wl, wr);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          atomicAdd(g1 + j * (2 * kNuCopies), nu_term(c1, wl[j], j < kNuSmall));
          atomicAdd(g2 + j * (2 * kNuCopies), nu_term(c2, wl[j], j < kNuSmall));
          atomicAdd(g1 + (7 - j) * (2 * kNuCopies), nu_term(c1, wr[j], j < kNuSmall));
          atomicAdd(g2 + (7 - j) * (2 * kNuCopies), nu_term(c2, wr[j], j < kNuSmall));
        }
      }
      if (!kBlocks || !blocks) load(c0);  // in flight while this turn is added up
      __syncthreads();
      // Add the turn up: half-warp h takes the octets of points o = h mod 16, which records
      // of the cells of octets o - 1 and o reach, one thread per point and part.
      const unsigned m0 = __ballot_sync(0xffffffffu, fl[lane] != 0), m1 = __ballot_sync(0xffffffffu, fl[32 + lane] != 0);
      const unsigned long long cells = (unsigned long long)m1 << 32 | m0, lit = cells | cells << 1;
#pragma unroll
      for (int r = 0; r < kNuBlock / 8 / 16 + 1; ++r) {
        const int o = r * 16 + (tid >> 4);
        const bool on = o < 64 ? (lit >> (o & 63)) & 1ull : o == 64 && (cells >> 63) != 0ull;
        if (!on) continue;
        const int i = o * 16 + (tid & 15);  // point i / 2, part i & 1
        const long long t = nu_add_up(nsm, i * (kNuCopies / 4), i >> 1);
        sum[i] = fmaf((float)t * cls.less, cls.down, sum[i]);
      }
      ++pass;
      if (kBlocks && blocks) __syncthreads();  // before the next block's additions (else: the next turn's barrier)
    }
  }
  bad = __syncthreads_or(bad);
  if (kBlocks) {
    store_block();
  } else {  // the points past the grid's end fold back
    for (int i = tid; i < M; i += kNuThreads) {
      float re = sum[2 * i], im = sum[2 * i + 1];
      for (int k = i + M; k < npts; k += M) {
        re += sum[2 * k];
        im += sum[2 * k + 1];
      }
      out[(i - (kNuW / 2 - 1)) & (M - 1)] = make_float2(re, im);
    }
  }
  if (bad) {
    __syncthreads();
    for (int i = tid; i < M; i += kNuThreads) out[i] = make_float2(NAN, NAN);
  }
}

// The split phase of a moving scene: CTA (q, v) spreads its records for the launch's
// chirps, up to kTile, a block of cells at a time (kBlocks: two, 512 samples).  From one
// chirp to the next a record's phasor turns by a constant and its grid position moves by
// a constant, so the preparation (two sines, the split phase) is paid once per tile, from
// that chirp's own delays, and a chirp costs a complex product and the sixteen additions:
// 12 antennas x 367,500 records x 128 chirps 3.5 ms against 5.0 in groups chirp by chirp
// (8 chirps at a time 3.9, 4 at a time 4.6; a third of it adds the chunks' copies up), 512
// samples, 12 x 8,600 records 843 -> 560 us.  The rounding of up to kTile - 1 turns adds
// 3e-7 to 7e-7 to the last chirp's error.  A chunk's sums go to the chirp's grid in global
// memory (L2), each point by one thread; kTile copies in shared memory would cost a
// resident CTA.
constexpr int kTile = 16;  // chirps per launch
template <bool kBlocks>
__global__ void __launch_bounds__(kNuThreads, 3)
    k_nufft_spread_chirps(const float4* __restrict__ prep, const float* __restrict__ rate, int64_t cap,
                          const int32_t* __restrict__ d_P, const NufftArg na, const __grid_constant__ NufftCoef co,
                          float2* __restrict__ grids) {
  extern __shared__ uint4 nsm[];  // [npts][re, im][kNuCopies]
  __shared__ uint32_t s_max[2];  // by the parity of the turn: largest amplitude
  __shared__ int s_log[2], s_pow[2];  // and the sums of the amplitudes' logarithms and, rarely, powers
  __shared__ int flag[2][kNuBlock / 8];
  const int M = 1 << na.log_m, bs = nu_cells(M), npts = nu_points(M), oct = bs >> 3;
  const int tid = threadIdx.x, lane = tid & 31;
  const int v = blockIdx.x % na.V, q = blockIdx.x / na.V, nc = na.chirps;
  float2* out = grids + (size_t)(q * na.V + v) * nc * M;
  for (int i = tid; i < npts * (2 * kNuCopies / 4); i += kNuThreads) nsm[i] = nu_zero();
  for (int i = tid; i < 2 * (kNuBlock / 8); i += kNuThreads) (&flag[0][0])[i] = 0;
  if (tid < 2) s_max[tid] = 0u, s_log[tid] = s_pow[tid] = 0;
  after_previous();
  for (int i = tid; i < nc * M; i += kNuThreads) out[i] = make_float2(0.f, 0.f);
  const int64_t P = *d_P;
  const int64_t r0 = P * q / na.Q;
  const int n = (int)(P * (q + 1) / na.Q - r0);
  const size_t at = (size_t)v * cap + r0;
  const bool upper = lane >= 16;
  int* mine = reinterpret_cast<int*>(nsm) + (lane & 15);
  int pass = 0;
  bool bad = false;  // a record that is not finite: the antenna's samples are NaN
  __syncthreads();
  bool again = false;
  int ceil = 0, left = min(kNuChunk, n);  // classes in turns, as k_nufft_spread
  for (int c0 = 0, chunk = 0; c0 < n; ++chunk) {
    float c1[kNuItems], c2[kNuItems], wr[kNuItems], wi[kNuItems], s[kNuItems], ds[kNuItems];
    int cell[kNuItems], logs = 0;
    uint32_t am = 0, mag[kNuItems];  // mag: the amplitudes' bits
#pragma unroll
    for (int u = 0; u < kNuItems; ++u) {
      const int p = c0 + tid + u * kNuThreads;
      float4 r = p < n ? __ldg(&prep[at + p]) : make_float4(0.f, 0.f, 0.f, 0.f);
      const float ld = p < n ? __ldg(&rate[at + p]) : 0.f;
      shift_record(r, ld, na.cyc0, na.eps0);  // the tile's first chirp
      float x = na.half_n * r.y;  // exact
      x -= rintf(x);
      x = fmaf(na.half_n, r.z, x) + r.x;
      const float uh = na.m * r.y;  // exact
      float fl = floorf(uh);
      float t = fmaf(na.m, r.z, uh - fl);
      int ce = (int)fl;
      bad |= !isfinite(x + t + r.w + ld);
      fl = floorf(t);
      s[u] = (t - fl) - 0.5f;
      cell[u] = (ce + (int)fl) & (M - 1);
      ds[u] = ld * na.move;
      float sn, cs;
      sincospif(2.f * x, &sn, &cs);
      // the lower half of a warp adds real parts first, the upper imaginary ones: with the turn's
      // sine negated, the swapped pair turns by the same formula
      c1[u] = r.w * (upper ? sn : cs);
      c2[u] = r.w * (upper ? cs : sn);
      sincospif(2.f * cycles_of(ld, na.turn), &sn, &cs);
      wr[u] = cs;
      wi[u] = upper ? -sn : sn;
      mag[u] = __float_as_uint(fabsf(r.w));
    }
    if (again) {
#pragma unroll
      for (int u = 0; u < kNuItems; ++u)
        if ((int)(mag[u] >> 20) >= ceil) c1[u] = c2[u] = 0.f, mag[u] = 0u;
    }
#pragma unroll
    for (int u = 0; u < kNuItems; ++u) {
      am = max(am, mag[u]);
      logs += (int)(mag[u] >> 20);
    }
    am = __reduce_max_sync(0xffffffffu, am);
    logs = __reduce_add_sync(0xffffffffu, logs);
    if (lane == 0) {
      atomicMax(&s_max[chunk & 1], am);
      atomicAdd(&s_log[chunk & 1], logs);
    }
    __syncthreads();
    logs = s_log[chunk & 1];
    const uint32_t top = s_max[chunk & 1];
    NuClass cls = nu_class(top, logs, left);
    again = false;
    if (__any_sync(0xffffffffu, cls.rare)) {  // the same for the whole CTA
      nu_rare(cls, top, logs, left);
      if (cls.floor) {
        float x = 0.f;
#pragma unroll
        for (int u = 0; u < kNuItems; ++u) {
          const float y = nu_part(__uint_as_float(mag[u]), cls);
          x = fmaf(y, y, x);
        }
        const int power = __reduce_add_sync(0xffffffffu, (int)x);
        if (lane == 0) atomicAdd(&s_pow[chunk & 1], power);
        __syncthreads();
        if (nu_one_class(cls, top, s_pow[chunk & 1], logs, left)) cls.floor = 0;
      }
      again = __any_sync(0xffffffffu, cls.floor != 0);
      ceil = cls.floor;
      if (again || cls.more != 1.f) {
#pragma unroll
        for (int u = 0; u < kNuItems; ++u) {
          const bool in = (int)(mag[u] >> 20) >= cls.floor;
          if (again) left -= __syncthreads_count(in);
          c1[u] = in ? c1[u] * cls.more : 0.f;
          c2[u] = in ? c2[u] * cls.more : 0.f;
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kNuItems; ++u) {
      c1[u] *= cls.up;
      c2[u] *= cls.up;
    }
    c0 += again ? 0 : kNuChunk;
    left = again ? left : min(kNuChunk, n - c0);
    // the turn before's words: read before this turn's first barrier
    if (tid == 0) s_max[~chunk & 1] = 0u, s_log[~chunk & 1] = s_pow[~chunk & 1] = 0;
    for (int kb = 0, b = 0; kb < (kBlocks ? nc * (M / bs) : nc); ++kb, ++pass) {
      const int k = kBlocks ? kb / (M / bs) : kb;
      if (kBlocks) b = kb - k * (M / bs);
      int* fl = flag[pass & 1];
      if (tid < kNuBlock / 8) flag[~pass & 1][tid] = 0;  // read before this pass
#pragma unroll
      for (int u = 0; u < kNuItems; ++u) {
        const int idx = kBlocks ? cell[u] - b * bs : cell[u];
        if ((!kBlocks || (unsigned)idx < (unsigned)bs) && (c1[u] != 0.f || c2[u] != 0.f)) {
          int* g1 = mine + idx * (2 * kNuCopies) + (upper ? kNuCopies : 0);
          int* g2 = mine + idx * (2 * kNuCopies) + (upper ? 0 : kNuCopies);
          fl[idx >> 3] = 1;
          float wl[4], wrt[4];
          nu_weights(co, s[u], wl, wrt);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            atomicAdd(g1 + j * (2 * kNuCopies), nu_term(c1[u], wl[j], j < kNuSmall));
            atomicAdd(g2 + j * (2 * kNuCopies), nu_term(c2[u], wl[j], j < kNuSmall));
            atomicAdd(g1 + (7 - j) * (2 * kNuCopies), nu_term(c1[u], wrt[j], j < kNuSmall));
            atomicAdd(g2 + (7 - j) * (2 * kNuCopies), nu_term(c2[u], wrt[j], j < kNuSmall));
          }
        }
        if (kBlocks && (b + 1) * bs < M) continue;
        // the next chirp
        const float a = c1[u];
        c1[u] = fmaf(a, wr[u], -c2[u] * wi[u]);
        c2[u] = fmaf(c2[u], wr[u], a * wi[u]);
        const float sh = s[u] + ds[u], f = floorf(sh + 0.5f);
        s[u] = sh - f;
        cell[u] = (cell[u] + (int)f) & (M - 1);
      }
      __syncthreads();
      // half-warp h adds up the octets of points o = h mod 16 (as k_nufft_spread), into the
      // chirp's grid; the points past the grid's end belong to octet 0, those past a block's
      // end to the next block, whose turn is another pass
      const unsigned m0 = __ballot_sync(0xffffffffu, fl[lane] != 0), m1 = __ballot_sync(0xffffffffu, fl[32 + lane] != 0);
      const unsigned long long cells = (unsigned long long)m1 << 32 | m0, last = kBlocks ? 0ull : cells >> (oct - 1) & 1ull,
                               lit = cells | cells << 1 | last;
      float* to = reinterpret_cast<float*>(out + (size_t)k * M);
#pragma unroll
      for (int r = 0; r < kNuBlock / 8 / 16 + (kBlocks ? 1 : 0); ++r) {
        const int o = r * 16 + (tid >> 4);
        if (kBlocks ? o > 64 || !(o < 64 ? lit >> o & 1ull : cells >> 63) : o >= oct || !((lit >> o) & 1ull)) continue;
        const int i = o * 16 + (tid & 15);  // point i / 2, part i & 1
        float* g = to + 2 * ((b * bs + (i >> 1) - (kNuW / 2 - 1)) & (M - 1)) + (i & 1);
        const float old = *g;
        long long t = nu_add_up(nsm, i * (kNuCopies / 4), i >> 1);
        if (!kBlocks && o == 0) t += nu_add_up(nsm, (i + 2 * M) * (kNuCopies / 4), (i >> 1) + M);
        *g = fmaf((float)t * cls.less, cls.down, old);
      }
      __syncthreads();
    }
  }
  bad = __syncthreads_or(bad);
  if (bad)
    for (int i = tid; i < nc * M; i += kNuThreads) out[i] = make_float2(NAN, NAN);
}

// Finishing, kNuFinSlice grid points per CTA: CTA (row, s) adds slice s of the Q
// CTAs' grids of a row (antenna and chirp) in a fixed order (kNuFinThreads / slice
// threads per point, each over every such CTA with four interleaved sums, then the
// threads' sums in order) into bsum; the last CTA of the row to finish (a counter
// per row, zeroed by the spreading kernel) runs the M-point FFT and the division
// by Psi(n'/M) and writes S[v][n] into the cube: the row's chirp of a moving scene,
// else every chirp (a static scene's chirps are equal).
constexpr int kNuFinThreads = 1024;
constexpr int kNuFinSlice = 128;
__global__ void __launch_bounds__(kNuFinThreads) k_nufft_finish(const float2* __restrict__ grids, const NufftArg na,
                                                                const __grid_constant__ NufftCoef co,
                                                                float2* __restrict__ bsum,
                                                                unsigned int* __restrict__ cnt,
                                                                float2* __restrict__ cube, int C, bool moving) {
  after_previous();
  next_may_start();
  extern __shared__ float2 sg[];  // slots(M) grid, slots(M / 2) twiddles, [kNuFinThreads] per-thread sums
  __shared__ int s_last;
  const int log_m = na.log_m, M = 1 << log_m, slice = M < kNuFinSlice ? M : kNuFinSlice, S = M / slice;
  const int row = blockIdx.x / S, sl = blockIdx.x - row * S, rows = na.V * na.chirps, Q = na.Q;
  float2* tw = sg + fft::slots(M);
  float2* part = tw + fft::slots(M / 2);
  const int parts = blockDim.x / slice, li = threadIdx.x % slice, k0 = threadIdx.x / slice;
  const int l = sl * slice + li;
  float2 a0 = make_float2(0.f, 0.f), a1 = a0, a2 = a0, a3 = a0;
  const float2* src = grids + (size_t)row * M + l;
  const size_t qs = (size_t)rows * M;  // from one CTA's grid to the next
  int q = k0;
  for (; q + 3 * parts < Q; q += 4 * parts) {  // four loads in flight, four interleaved sums
    const float2 x0 = __ldcg(src + (size_t)q * qs), x1 = __ldcg(src + (size_t)(q + parts) * qs);
    const float2 x2 = __ldcg(src + (size_t)(q + 2 * parts) * qs), x3 = __ldcg(src + (size_t)(q + 3 * parts) * qs);
    a0.x += x0.x;
    a0.y += x0.y;
    a1.x += x1.x;
    a1.y += x1.y;
    a2.x += x2.x;
    a2.y += x2.y;
    a3.x += x3.x;
    a3.y += x3.y;
  }
  for (; q < Q; q += parts) {
    const float2 x = __ldcg(src + (size_t)q * qs);
    a0.x += x.x;
    a0.y += x.y;
  }
  part[threadIdx.x] = make_float2((a0.x + a1.x) + (a2.x + a3.x), (a0.y + a1.y) + (a2.y + a3.y));
  __syncthreads();
  if (threadIdx.x < slice) {
    float2 acc = part[li];
    for (int k = 1; k < parts; ++k) {
      acc.x += part[k * slice + li].x;
      acc.y += part[k * slice + li].y;
    }
    bsum[(size_t)row * M + l] = acc;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&cnt[row], 1u) == (unsigned)(S - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  fft::fill_twiddles(tw, M, 1.f, blockDim.x, threadIdx.x);
  for (int i = threadIdx.x; i < M; i += blockDim.x) sg[fft::slot(fft::bitrev(i, log_m))] = __ldcg(&bsum[(size_t)row * M + i]);
  __syncthreads();
  fft::smem_fft(sg, tw, log_m, blockDim.x, threadIdx.x);
  const int Ns = M >> 1, h = Ns >> 1;
  // rows are (antenna, chirp of the launch), the chirp fastest
  const int v = row / na.chirps;
  const int c0 = moving ? na.chirp0 + row - v * na.chirps : 0, c1 = moving ? c0 + 1 : C;
  for (int n = threadIdx.x; n < Ns; n += blockDim.x) {
    const float xi = (float)(n - h) / (float)h, y = xi * xi;
    float inv = co.inv[8];
#pragma unroll
    for (int k = 7; k >= 0; --k) inv = fmaf(inv, y, co.inv[k]);
    const float2 B = sg[fft::slot((n - h) & (M - 1))];
    const float2 val = make_float2(B.x * inv, B.y * inv);
    for (int c = c0; c < c1; ++c) cube[((size_t)v * C + c) * Ns + n] = val;
  }
}

// Finishing of grids of up to kNuClusterPoints points: a cluster of eight CTAs per row.
// CTA r adds the r-th eighth of the Q grids (as many threads per point as there are,
// then the threads' sums in order), the CTAs exchange their eighths through each
// other's shared memory, and each that has chirps of the row to write transforms the
// whole grid (three or four passes: cheaper than handing the result on) and writes
// its share of them.  A chain of latencies, so it is the links that count: no partial
// sums through L2, no fence and counter, a static scene's chirps written by 8 V CTAs
// instead of V (12 antennas x 128 chirps x 256 samples: about 10 -> 6 us).
// Above 1024 points a CTA's eighth leaves too few threads per point for the grids' sum
// (2048 points: 109 us for a synthesis that takes 105 with the kernel above).
constexpr int kNuClusterPoints = 1024;
constexpr int kNuRanks = 8;
constexpr int kNuClThreads = 512;
__global__ void __cluster_dims__(kNuRanks, 1, 1) __launch_bounds__(kNuClThreads)
    k_nufft_finish_cluster(const float2* __restrict__ grids, const NufftArg na, const __grid_constant__ NufftCoef co,
                           float2* __restrict__ cube, int C, bool moving) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ float2 sg[];  // slots(M) grid, slots(M / 2) twiddles, [kNuClThreads] per-thread sums, [M / 8] this eighth
  const int log_m = na.log_m, M = 1 << log_m, pts = M / kNuRanks, rank = (int)cluster.block_rank();
  const int row = blockIdx.x / kNuRanks, rows = na.V * na.chirps, Q = na.Q, tid = threadIdx.x;
  float2* tw = sg + fft::slots(M);
  float2* part = tw + fft::slots(M / 2);
  float2* mine = part + kNuClThreads;
  const int parts = kNuClThreads / pts, li = tid % pts, k0 = tid / pts;  // pts <= 128
  const float2* src = grids + (size_t)row * M + rank * pts + li;
  const size_t qs = (size_t)rows * M;  // from one CTA's grid to the next
  // this CTA's chirps of the row (of a moving scene's one chirp: all of it to CTA 0)
  const int c0 = moving ? (rank == 0 ? 0 : 1) : C * rank / kNuRanks, c1 = moving ? 1 : C * (rank + 1) / kNuRanks;
  if (c0 < c1) fft::fill_twiddles(tw, M, 1.f, kNuClThreads, tid);
  after_previous();
  next_may_start();
  float2 a0 = make_float2(0.f, 0.f), a1 = a0, a2 = a0, a3 = a0;
  int q = k0;
  for (; q + 3 * parts < Q; q += 4 * parts) {  // four loads in flight, four interleaved sums
    const float2 x0 = __ldcg(src + (size_t)q * qs), x1 = __ldcg(src + (size_t)(q + parts) * qs);
    const float2 x2 = __ldcg(src + (size_t)(q + 2 * parts) * qs), x3 = __ldcg(src + (size_t)(q + 3 * parts) * qs);
    a0 = make_float2(a0.x + x0.x, a0.y + x0.y);
    a1 = make_float2(a1.x + x1.x, a1.y + x1.y);
    a2 = make_float2(a2.x + x2.x, a2.y + x2.y);
    a3 = make_float2(a3.x + x3.x, a3.y + x3.y);
  }
  for (; q < Q; q += parts) {
    const float2 x = __ldcg(src + (size_t)q * qs);
    a0 = make_float2(a0.x + x.x, a0.y + x.y);
  }
  part[tid] = make_float2((a0.x + a1.x) + (a2.x + a3.x), (a0.y + a1.y) + (a2.y + a3.y));
  __syncthreads();
  if (tid < pts) {
    float2 acc = part[tid];
    for (int k = 1; k < parts; ++k) acc = make_float2(acc.x + part[k * pts + tid].x, acc.y + part[k * pts + tid].y);
    mine[tid] = acc;
  }
  cluster.sync();
  if (c0 < c1) {
    for (int i = tid; i < M; i += kNuClThreads)
      sg[fft::slot(fft::bitrev(i, log_m))] = cluster.map_shared_rank(mine, i / pts)[i % pts];
  }
  cluster.sync();  // every eighth has been read: a CTA may leave
  if (c0 >= c1) return;
  fft::smem_fft(sg, tw, log_m, kNuClThreads, tid);
  // rows are (antenna, chirp of the launch), the chirp fastest
  const int Ns = M >> 1, h = Ns >> 1, v = row / na.chirps, first = moving ? na.chirp0 + row - v * na.chirps : c0;
  const int last = moving ? first + 1 : c1;
  // threads over samples, then over chirps; one 8-byte store each (a cube need not be
  // aligned to more)
  float2* out = cube + (size_t)v * C * Ns;
  const int groups = kNuClThreads / Ns > 0 ? kNuClThreads / Ns : 1, g = tid / Ns;
  for (int n = tid % Ns; n < Ns && g < groups; n += kNuClThreads) {
    const float xi = (float)(n - h) / (float)h, y = xi * xi;
    float inv = co.inv[8];
#pragma unroll
    for (int k = 7; k >= 0; --k) inv = fmaf(inv, y, co.inv[k]);
    const float2 B = sg[fft::slot((n - h) & (M - 1))];
    const float2 val = make_float2(B.x * inv, B.y * inv);
    for (int c = first + g; c < last; c += groups) out[(size_t)c * Ns + n] = val;
  }
}

double bessel_i0(double x) { return bessel_i0_of(0.25 * x * x); }

double kb_kernel(double x) {
  const double z = 2.0 * x / kNuW, y = 1.0 - z * z;
  return y > 0.0 ? bessel_i0(kNuBeta * sqrt(y)) / bessel_i0(kNuBeta) : (y < 0.0 ? 0.0 : 1.0 / bessel_i0(kNuBeta));
}

// Monomial coefficients of the degree-n interpolant of f at the Chebyshev nodes of
// [0, b] (Newton's divided differences, expanded).
template <int n, class F>
void fit_poly(F f, double b, float* out) {
  double x[n + 1], d[n + 1], m[n + 1] = {};
  for (int i = 0; i <= n; ++i) {
    x[i] = 0.5 * b * (1.0 + cos(M_PI * (i + 0.5) / (n + 1)));
    d[i] = f(x[i]);
  }
  for (int k = 1; k <= n; ++k)
    for (int i = n; i >= k; --i) d[i] = (d[i] - d[i - 1]) / (x[i] - x[i - k]);
  for (int k = n; k >= 0; --k) {  // m <- m (x - x_k) + d_k
    for (int i = n; i >= 1; --i) m[i] = m[i - 1] - x[k] * m[i];
    m[0] = -x[k] * m[0] + d[k];
  }
  for (int i = 0; i <= n; ++i) out[i] = (float)m[i];
}

NufftCoef make_nufft_coef() {
  NufftCoef c{};
  for (int j = 0; j < 4; ++j) {  // the even and odd parts of psi_j in y = s^2
    const double a = j - 0.5 * (kNuW - 1);
    float e[5], o[4];
    fit_poly<4>([&](double y) { return 0.5 * (kb_kernel(a - sqrt(y)) + kb_kernel(a + sqrt(y))); }, 0.25, e);
    fit_poly<3>([&](double y) { return 0.5 * (kb_kernel(a - sqrt(y)) - kb_kernel(a + sqrt(y))) / sqrt(y); }, 0.25, o);
    for (int k = 0; k < 5; ++k) c.e[k][j] = e[k];
    for (int k = 0; k < 4; ++k) c.o[k][j] = o[k];
  }
  // Psi(xi) = w / I0(beta) sinh(r) / r, r = sqrt(beta^2 - (pi w xi)^2), real on the band
  // |xi| <= 1/4; its reciprocal in y = (4 xi)^2 = (2 n' / N_s)^2
  fit_poly<8>(
      [&](double y) {
        const double a = M_PI * kNuW * 0.25, r = sqrt(kNuBeta * kNuBeta - a * a * y);
        return bessel_i0(kNuBeta) * r / (kNuW * sinh(r));
      },
      1.0, c.inv);
  return c;
}

const NufftCoef& nufft_coef() {
  static const NufftCoef c = make_nufft_coef();
  return c;
}

// ---- adjoint by the type-2 non-uniform FFT ----------------------------------
//
// Eq. 11-12 need, per (path, antenna), sums over the samples of the upstream
// gradient against the path's phasors.  With h[n'] = conj(g[n' + N_s/2]) and
// e^{j 2 pi x}, x = phi0 + (N_s/2) delta, the phasor at n' = 0,
//   Z0 = e^{j 2 pi x} sum_n' h[n'] e^{j 2 pi n' delta},            dL/dA = Re Z0,
//   Z1 = the same sum with weights 1 + (n' + N_s/2) B / (f_c N_s),  dL/dL = -2 pi A f_c / c Im Z1,
// and dL/d(phase offset) = -2 pi A Im Z0.  Both sums are band-limited functions of
// delta, so they are read off a grid of M = 2 N_s points (one M-point FFT each of
// h / Psi(n'/M)) with the spreading kernel's eight weights: a path costs eight
// 16-byte reads and 32 FMAs instead of N_s phasors and 6 N_s FMAs.  12 antennas x
// 367,500 paths x 256 samples, 128 chirps: 43 us (505 us term by term), 16 us of them
// the records' 16 bytes in and 8 out at the copy rate; error against FP64 2.8e-7
// (6.8e-7).

constexpr int kAdjThreads = 512;
constexpr int kAdjMargin = kNuW;  // the grid is stored with its wrap-around: entry i is point i - 3

// One cluster per antenna: its CTAs sum a share of the chirps each (a static scene's
// chirps see the same paths), CTAs 0 and 1 then transform Z0's and Z1's coefficients
// and write their halves of the grid's float4 entries.
__global__ void __launch_bounds__(kAdjThreads) k_adj_grid(const float2* __restrict__ g, int V, int C, int Ns, int log_m,
                                                          float slope, const __grid_constant__ NufftCoef co,
                                                          float2* __restrict__ out) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ float2 sa[];  // [N_s] this CTA's chirps summed, slots(M) grid, slots(M / 2) twiddles
  const int M = 1 << log_m, rank = (int)cluster.block_rank(), ranks = (int)cluster.num_blocks();
  const int v = blockIdx.x / ranks, h = Ns >> 1;
  float2* s = sa + Ns;
  float2* tw = s + fft::slots(M);
  const int c0 = C * rank / ranks, c1 = C * (rank + 1) / ranks;
  if (rank < 2) {
    fft::fill_twiddles(tw, M, 1.f, kAdjThreads, threadIdx.x);
    for (int i = threadIdx.x; i < fft::slots(M); i += kAdjThreads) s[i] = make_float2(0.f, 0.f);
  }
  after_previous();
  next_may_start();
  for (int n = threadIdx.x; n < Ns; n += kAdjThreads) {
    float2 a = make_float2(0.f, 0.f);
#pragma unroll 8
    for (int c = c0; c < c1; ++c) {
      const float2 x = __ldg(&g[((size_t)v * C + c) * Ns + n]);
      a.x += x.x;
      a.y += x.y;
    }
    sa[n] = a;
  }
  cluster.sync();
  if (rank < 2) {
    for (int n = threadIdx.x; n < Ns; n += kAdjThreads) {
      float2 a = make_float2(0.f, 0.f);
      for (int r = 0; r < ranks; ++r) {
        const float2 x = cluster.map_shared_rank(sa, r)[n];
        a.x += x.x;
        a.y += x.y;
      }
      const float xi = (float)(n - h) / (float)h, y = xi * xi;
      float w = co.inv[8];
#pragma unroll
      for (int k = 7; k >= 0; --k) w = fmaf(w, y, co.inv[k]);
      if (rank == 1) w *= fmaf((float)n, slope, 1.f);
      s[fft::slot(fft::bitrev((n - h) & (M - 1), log_m))] = make_float2(a.x * w, -a.y * w);
    }
    __syncthreads();
    fft::smem_fft(s, tw, log_m, kAdjThreads, threadIdx.x);
    float2* o = out + 2 * (size_t)v * (M + kAdjMargin) + rank;
    for (int i = threadIdx.x; i < M + kAdjMargin; i += kAdjThreads) o[2 * i] = s[fft::slot((i - (kNuW / 2 - 1)) & (M - 1))];
  }
  cluster.sync();  // no CTA leaves while another may read its shared memory
}

// One record per thread at a time, the grid's CTAs striding over antenna blockIdx.y's
// records.  The grid (8 KB to 131 KB per antenna) is read through L1, where the
// neighbouring rays of a warp share lines.
__global__ void __launch_bounds__(256) k_synth_bwd_nufft(const float4* __restrict__ prep, int64_t cap,
                                                         const int32_t* __restrict__ d_P, int log_m,
                                                         const __grid_constant__ NufftCoef co,
                                                         const float4* __restrict__ grid, float inv_lambda,
                                                         float* __restrict__ glen, float* __restrict__ gamp,
                                                         float* __restrict__ gphase) {
  after_previous();
  const int v = blockIdx.y, M = 1 << log_m, P = *d_P;
  const float m = (float)M, half_n = 0.25f * m;
  const size_t row = (size_t)v * cap;
  const float4* gv = grid + (size_t)v * (M + kAdjMargin);
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < P; p += (int64_t)gridDim.x * blockDim.x) {
    const float4 r = __ldg(&prep[row + p]);
    float x = half_n * r.y;  // exact
    x -= rintf(x);
    x = fmaf(half_n, r.z, x) + r.x;
    const float uh = m * r.y;  // exact
    float fl = floorf(uh);
    float t = fmaf(m, r.z, uh - fl);
    int cell = (int)fl;
    fl = floorf(t);
    t -= fl;
    cell = (cell + (int)fl) & (M - 1);
    float wl[4], wr[4];
    nu_weights(co, t - 0.5f, wl, wr);
    float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    auto add = [&](float w, float4 q) {
      z.x = fmaf(w, q.x, z.x);
      z.y = fmaf(w, q.y, z.y);
      z.z = fmaf(w, q.z, z.z);
      z.w = fmaf(w, q.w, z.w);
    };
#pragma unroll
    for (int j = 0; j < 4; ++j) {  // outermost points first: the smallest weights
      add(wl[j], __ldg(&gv[cell + j]));
      add(wr[j], __ldg(&gv[cell + 7 - j]));
    }
    float sn, cs;
    sincospif(2.f * x, &sn, &cs);
    gamp[row + p] = cs * z.x - sn * z.y;
    glen[row + p] = -kTwoPiF * r.w * inv_lambda * (cs * z.w + sn * z.z);
    if (gphase) gphase[row + p] = -kTwoPiF * r.w * (cs * z.y + sn * z.x);
  }
}

inline size_t adj_smem(int Ns) { return sizeof(float2) * (size_t)(Ns + fft::slots(2 * Ns) + fft::slots(Ns)); }

cudaError_t adj_attr(int Ns) {
  static std::atomic<uint64_t> done{0};  // bit per device ordinal below 64
  if (adj_smem(Ns) <= 48 * 1024) return cudaSuccess;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 64 && ((done.load() >> dev) & 1u)) return cudaSuccess;
  e = cudaFuncSetAttribute(k_adj_grid, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)adj_smem(4096));
  if (e == cudaSuccess && dev < 64) done.fetch_or(1ull << dev);
  return e;
}

// When the grids beat the direct kernel (k_chirp_sum, k_synth_bwd), by record slots
// (path_cap x antennas), measured: 256 samples, one chirp, 6.9 against 6.5 us at
// 32,768 and 7.0 against 10.4 us at 64,800; 64 samples 6.5 against 4.3 us at 131,072
// and 7.2 against 9.1 us at 524,288; 1024 samples 12.1 against 14.0 us at 512
// already; 128 chirps (whose sum the direct kernel's one CTA per antenna waits for)
// 9.3 against 11.4 us at 1,536.
inline bool adj_nufft_for(int Ns, int C, int64_t records) {
  return Ns >= 1024 || C >= 8 || records * Ns >= (3 << 22);
}

// Few (path, antenna) record slots: the direct kernels, whose one pass over the
// records costs less than the non-uniform FFT's spreading, finishing sum and FFT
// chain.  Measured crossings (4 antennas, one wave of either): up to 512 samples,
// where the tensor-core kernel sums directly, 8.5-10 us against 9-14 us at 32,768
// slots, 11-12 against 11-14 us at 73,728, 23 against 13-15 us at 262,088; above,
// 10-26 against 17-41 us at 2,048 slots, 19-59 against 17-47 us at 8,192.
constexpr int kNuMovingMaxSamples = 512;  // the split phase of a moving scene
// The FP64 phase always goes to the non-uniform FFT, which forms each path's carrier
// phase and grid position in FP64 and leaves no per-sample FP64 work: 13-46 us
// against 32-248 us at 512 slots and 64-4096 samples, 29 us against 2.64 ms at
// 524,288 and 1024, and 1.0-2.6e-7 from FP64 against 3.3e-7-2.7e-6 (the term-by-term
// kernel's FP32 sums).
inline bool nufft_for(sbr_phase_mode mode, int Ns, int64_t records) {
  if (mode == SBR_PHASE_FP64) return true;
  return mode == SBR_PHASE_SPLIT && records >= (Ns <= 512 ? 65536 : 8192);
}

// Launch-shape queries are cached per device ordinal (kernel attributes such as
// a raised shared-memory limit are per device too); ordinals at or beyond
// kDevCache are queried on every call.
constexpr int kDevCache = 64;

inline int current_device() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) dev = 0;
  return dev;
}

// Grid: V * Q CTAs, Q the largest that keeps every CTA resident at once (one
// wave), capped by the number of path chunks.
// dynamic shared memory of the split kernel: the groups' reduction buffer
inline size_t split_smem(int Ns) {
  const int T = threads_for(Ns), M = Ns / T;
  return kSplitThreads / T > 1 ? sizeof(float2) * M * kSplitThreads : 0;
}

// resident CTAs of the split kernel per SM (registers and shared memory decide)
int split_per_sm(int Ns) {
  static int cache[kDevCache][17] = {};
  const int T = threads_for(Ns), M = Ns / T;
  if (M > 16) return 1;
  const int dev = current_device();
  if (dev < kDevCache && cache[dev][M]) return cache[dev][M];
  int n = 0;
  const size_t sm = split_smem(Ns);
  switch (M) {
    case 1: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_synth_split<1>, kSplitThreads, sm); break;
    case 2: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_synth_split<2>, kSplitThreads, sm); break;
    case 4: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_synth_split<4>, kSplitThreads, sm); break;
    case 8: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_synth_split<8>, kSplitThreads, sm); break;
    default: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_synth_split<16>, kSplitThreads, sm); break;
  }
  n = n > 0 ? n : 1;
  if (dev < kDevCache) cache[dev][M] = n;
  return n;
}

// resident CTAs of the tensor-core kernel per SM (N_s = 256 or 512)
int mma_per_sm(int Ns) {
  static int cache[kDevCache][3] = {};
  const int mt = Ns / 256;
  const int dev = current_device();
  if (dev < kDevCache && cache[dev][mt]) return cache[dev][mt];
  int n = 0;
  if (mt == 1) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_synth_mma<1>, kMmaThreads, 0);
  else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_synth_mma<2>, kMmaThreads, 0);
  n = n > 0 ? n : 1;
  if (dev < kDevCache) cache[dev][mt] = n;
  return n;
}

void grid_shape(int V, int Ns, int64_t cap, int* Q) {
  int per_sm = split_per_sm(Ns);
  if (Ns == 256 || Ns == 512) {
    const int m = mma_per_sm(Ns);
    if (m < per_sm) per_sm = m;
  }
  // whole waves only: every CTA resident from the start (a CTA beyond the
  // first wave would run alone after the others and double the launch)
  int64_t q = ((int64_t)sm_count() * per_sm) / V;
  const int64_t chunks = (cap + kChunk - 1) / kChunk;
  if (q > chunks) q = chunks;
  if (q < 1) q = 1;
  *Q = (int)q;
}

// dynamic shared memory of the spreading kernel: the grid's copies and its sums
inline size_t nufft_smem(int Ns) { return (2 * kNuCopies * sizeof(int) + 2 * sizeof(float)) * (size_t)nu_points(2 * Ns); }
inline auto chirps_kernel(int Ns) { return 2 * Ns > kNuBlock ? k_nufft_spread_chirps<true> : k_nufft_spread_chirps<false>; }
inline size_t nufft_chirps_smem(int Ns) { return 2 * kNuCopies * sizeof(int) * (size_t)nu_points(2 * Ns); }
inline size_t nufft_cl_smem(int Ns) {
  return sizeof(float2) * (size_t)(fft::slots(2 * Ns) + fft::slots(Ns) + kNuClThreads + 2 * Ns / kNuRanks);
}
inline size_t nufft_fin_smem(int Ns) { return sizeof(float2) * (size_t)(fft::slots(2 * Ns) + fft::slots(Ns) + kNuFinThreads); }

using NufftSpread = void (*)(const float4*, const float2*, const float*, const float*, int64_t, const int32_t*, NufftArg,
                             NufftCoef, float2*, unsigned int*);
template <bool kBlocks>
NufftSpread nufft_kernel_of(bool fp64, bool moving) {
  if (fp64) return moving ? k_nufft_spread<true, true, kBlocks> : k_nufft_spread<true, false, kBlocks>;
  return moving ? k_nufft_spread<false, true, kBlocks> : k_nufft_spread<false, false, kBlocks>;
}
inline NufftSpread nufft_kernel(int Ns, bool fp64, bool moving) {
  return 2 * Ns > kNuBlock ? nufft_kernel_of<true>(fp64, moving) : nufft_kernel_of<false>(fp64, moving);
}

constexpr int kMinSamples = 32, kMaxSamples = 4096;  // check_radar's

// resident spreading CTAs per SM (shared memory and registers decide); raises
// the kernels' shared-memory limits once where they pass 48 KB.  A limit belongs to
// the kernel, whatever the sample count it was raised for, and the counts are cached
// one by one: each is the most its kernel ever asks for, so none lowers another's.
int nufft_per_sm(int Ns) {
  static int cache[kDevCache][16] = {};
  int lg = 0;
  while ((1 << lg) < Ns) ++lg;
  const int dev = current_device();
  if (dev < kDevCache && cache[dev][lg]) return cache[dev][lg];
  const size_t sm = nufft_smem(Ns);
  int n = 32;
  for (int i = 0; i < 4; ++i) {
    const NufftSpread k = nufft_kernel(Ns, (i & 2) != 0, (i & 1) != 0);
    if (sm > 48 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    int m = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&m, k, kNuThreads, sm);
    n = std::min(n, m > 0 ? m : 1);
  }
  if (nufft_chirps_smem(Ns) > 48 * 1024)
    cudaFuncSetAttribute(chirps_kernel(Ns), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)nufft_chirps_smem(Ns));
  if (nufft_fin_smem(Ns) > 48 * 1024)
    cudaFuncSetAttribute(k_nufft_finish, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)nufft_fin_smem(kMaxSamples));
  if (dev < kDevCache) cache[dev][lg] = n;
  return n;
}

// CTAs per antenna of the spreading kernel: one wave, at most one per 256 paths
void nufft_shape(int V, int Ns, int64_t cap, int* Qn) {
  int64_t q = ((int64_t)sm_count() * nufft_per_sm(Ns)) / V;
  const int64_t batches = (cap + 255) / 256;
  if (q > batches) q = batches;
  if (q < 1) q = 1;
  *Qn = (int)q;
}

// Moving scenes whose chirps go in tiles: records enough to fill the CTAs that every launch
// of a tile puts to work, chirps enough to pay for the slower inner loop.  Tiles / groups:
// 12 antennas x 256 samples x 128 chirps, slots per antenna 4,050: 368 / 193 us, 7,200: 378 /
// 679; 4 antennas, 7,200: 273 / 113, 12,800: 284 / 398, 28,800: 300 / 635; 16 chirps, 12,800:
// 35 / 16, 28,800: 38 / 81; 2 chirps x 320,000: 20.7 / 17.3; 512 samples x 128 chirps, 4
// antennas, 28,800: 444 / 800.
constexpr int64_t kTileSlots = 65536;  // all antennas'
inline bool nufft_tiles(int V, int C, int Ns, int64_t cap) {
  return Ns <= kNuMovingMaxSamples && C >= 4 && V * cap >= kTileSlots;
}

// Grids per antenna in the workspace: one per spreading CTA, and for the chirps of a moving
// scene a tile's from each (at most 30 MB, 60 with 512 samples) or, in groups, a wave's (a
// group is then not held to the few CTAs that few paths ask for: 512 samples, 128 chirps x 950
// records 1.01 -> 0.13 ms).
inline int nufft_wave(int V, int qn, int C, int Ns) {
  return (int)std::max<int64_t>(qn, std::min<int64_t>((int64_t)qn * C, (int64_t)sm_count() * nufft_per_sm(Ns) / V));
}
inline int nufft_grids(int V, int qn, int C, int Ns, int64_t cap) {
  return nufft_tiles(V, C, Ns, cap) ? qn * std::min(C, kTile) : nufft_wave(V, qn, C, Ns);
}

// Summed grids per antenna: none where a cluster finishes the rows.
inline int nufft_sums(int rows, int Ns) { return 2 * Ns <= kNuClusterPoints ? 0 : rows; }

struct SynthWs {
  float2* partial;        // per-CTA partial sums of the direct kernels
  float2* gsum;           // chirp-summed upstream gradient of the adjoint
  float2* grids;          // non-uniform FFT: the CTAs' grids, V * Qg
  float2* bsum;           // non-uniform FFT: the rows' summed grids, nufft_sums
  unsigned int* fin_cnt;  // non-uniform FFT: finishing counters, V * rows
  float4* adj;            // adjoint: the antennas' grids
  int Q, Qn, Qg, rows;    // per antenna: CTAs (direct, FFT), grids, chirps that one launch may finish
};

// The workspace in `mem` (or its size alone) with room for the launches of `chirps`
// chirps of a moving scene.  One is all that a static scene and the adjoint use, and
// enough for a moving scene too, whose chirps then go one launch each.
size_t ws_layout(const sbr_radar_cfg* radar, int64_t cap, int chirps, void* mem, SynthWs* w) {
  const int V = radar->n_tx * radar->n_rx, Ns = radar->n_samples;
  grid_shape(V, Ns, cap, &w->Q);
  nufft_shape(V, Ns, cap, &w->Qn);
  w->Qg = nufft_grids(V, w->Qn, chirps, Ns, cap);
  w->rows = std::max(1, std::min(chirps, w->Qg));
  Carver c(mem);
  w->partial = c.take<float2>((size_t)V * w->Q * Ns);
  w->gsum = c.take<float2>((size_t)V * Ns);
  w->grids = c.take<float2>((size_t)V * w->Qg * 2 * Ns);
  w->bsum = c.take<float2>((size_t)V * nufft_sums(w->rows, Ns) * 2 * Ns);
  w->fin_cnt = c.take<unsigned int>((size_t)V * w->rows);
  w->adj = c.take<float4>((size_t)V * (2 * Ns + kAdjMargin));
  return c.bytes();
}

}  // namespace
}  // namespace sbr

using namespace sbr;

extern "C" size_t sbr_synth_ws_bytes(const sbr_radar_cfg* radar, int64_t path_cap) {
  if (!radar || radar->n_tx < 1 || radar->n_rx < 1) return 0;
  const int Ns = radar->n_samples;  // the layout asks the device about kernels that exist for these sizes alone
  if (Ns < kMinSamples || Ns > kMaxSamples || (Ns & (Ns - 1)) != 0) {
    set_error("sbr_synth_ws_bytes: n_samples=%d must be a power of two in [%d, %d]", Ns, kMinSamples, kMaxSamples);
    return 0;
  }
  SynthWs w;
  return ws_layout(radar, path_cap, radar->n_chirps, nullptr, &w);
}

namespace {
sbr_status bind_ws(const sbr_radar_cfg* radar, int64_t cap, bool moving, void* ws, size_t bytes, SynthWs* w,
                   const char* who) {
  SBR_ARG(ws && aligned256(ws), "%s: workspace NULL or not 256-byte aligned", who);
  if (moving && ws_layout(radar, cap, radar->n_chirps, ws, w) <= bytes) return SBR_OK;
  const size_t need = ws_layout(radar, cap, 1, ws, w);
  if (bytes < need) {
    set_error("%s: workspace of %zu bytes, %zu needed", who, bytes, need);
    return SBR_ERR_OOM;
  }
  return SBR_OK;
}

// The launch's constants; sets the kernels' shared-memory limits before their first launch.
NufftArg nufft_arg(const sbr_paths* p, const sbr_radar_cfg* r, int Q, int c0, int chirps) {
  const int Ns = r->n_samples, M = 2 * Ns;
  NufftArg na{};
  while ((1 << na.log_m) < M) ++na.log_m;
  na.half_n = 0.5f * (float)Ns;
  na.m = (float)M;
  na.f0_c = r->f0 / kC;
  na.b_cn = r->bandwidth / (kC * Ns);
  na.cyc = na.f0_c + 0.5 * Ns * na.b_cn;  // N_s / 2 is whole: delta need not be reduced first
  na.cell = M * na.b_cn;
  na.V = p->n_virt;
  na.Q = Q;
  na.chirps = chirps;
  na.chirp0 = c0;
  na.per_chirp = r->chirp_rep;
  na.cyc0 = Pair32(c0 * na.per_chirp * na.f0_c);
  na.eps0 = Pair32(c0 * na.per_chirp * na.b_cn);
  na.turn = Pair32(na.per_chirp * na.cyc);
  na.move = (float)(na.per_chirp * na.cell);
  nufft_per_sm(Ns);
  return na;
}

// The non-uniform FFT of chirps [c0, c0 + chirps) of a moving scene, or of a static
// scene's one chirp, written to all of them: spread by Q CTAs per antenna and chirp
// (Q * chirps <= w.Qg, chirps <= w.rows), then finish.
void launch_nufft(sbr_phase_mode mode, const sbr_paths* p, const sbr_radar_cfg* r, const SynthWs& w, bool moving, int Q,
                  int c0, int chirps, float2* cube, cudaStream_t st) {
  const int V = p->n_virt, Ns = r->n_samples, M = 2 * Ns;
  const NufftArg na = nufft_arg(p, r, Q, c0, chirps);
  const NufftCoef& co = nufft_coef();
  const float4* prep = reinterpret_cast<const float4*>(p->prep);
  const float2* plen = reinterpret_cast<const float2*>(p->path_len);
  const int grid = V * Q * chirps;
  ::sbr::note_launch();
  launch_after(nufft_kernel(Ns, mode == SBR_PHASE_FP64, moving), grid, kNuThreads, nufft_smem(Ns), st, prep, plen,
               p->phase_ofs, p->path_rate, p->path_cap, p->count, na, co, w.grids, w.fin_cnt);
  ::sbr::note_launch();
  if (M <= kNuClusterPoints) {
    launch_after(k_nufft_finish_cluster, V * chirps * kNuRanks, kNuClThreads, nufft_cl_smem(Ns), st, w.grids, na, co,
                 cube, r->n_chirps, moving);
    return;
  }
  const int slices = M / kNuFinSlice;
  launch_after(k_nufft_finish, V * chirps * slices, kNuFinThreads, nufft_fin_smem(Ns), st, w.grids, na, co, w.bsum,
               w.fin_cnt, cube, r->n_chirps, moving);
}

// The chirps of a moving scene, kTile at a time: a launch is one wave of CTAs, each with
// its share of the records and all chirps of the tile.
void launch_chirps(const sbr_paths* p, const sbr_radar_cfg* r, const SynthWs& w, float2* cube, cudaStream_t st) {
  const int V = p->n_virt, Ns = r->n_samples, C = r->n_chirps;
  for (int c = 0; c < C; c += kTile) {
    const NufftArg na = nufft_arg(p, r, w.Qn, c, std::min(kTile, C - c));
    ::sbr::note_launch();
    launch_after(chirps_kernel(Ns), V * w.Qn, kNuThreads, nufft_chirps_smem(Ns), st,
                 reinterpret_cast<const float4*>(p->prep), p->path_rate, p->path_cap, p->count, na, nufft_coef(), w.grids);
    ::sbr::note_launch();
    launch_after(k_nufft_finish_cluster, V * na.chirps * kNuRanks, kNuClThreads, nufft_cl_smem(Ns), st, w.grids, na,
                 nufft_coef(), cube, C, true);
  }
}

// A moving scene: every chirp synthesised from its own delays (split phase up to 512
// samples, or the FP64 phase), in tiles of chirps or (the FP64 phase, few records, few
// chirps) a group of chirps per launch.  A group's launch is one wave of Q
// CTAs per antenna and chirp; fewer CTAs per chirp mean fewer launches and the same
// records per CTA in all, so Q is the one whose launches / Q, the chirps' share of a
// wave each, is least (12 antennas x 128 chirps: 2 CTAs each, 7 launches of 19 chirps,
// 3.5 against the ideal 3.4; the records are then read from L2 by the chirps of a
// launch).  256 samples, 12 x 367,500 records x 128 chirps: 7.85 ms with one launch
// pair per chirp, 6.3 in groups (both before the leaner spreading; 5.0 after it).
sbr_status launch_moving(sbr_phase_mode mode, const sbr_paths* p, const sbr_radar_cfg* r, const SynthWs& w,
                         float2* cube, cudaStream_t st) {
  if (mode == SBR_PHASE_FP64 || (mode == SBR_PHASE_SPLIT && r->n_samples <= kNuMovingMaxSamples)) {
    const int C = r->n_chirps;
    if (mode == SBR_PHASE_SPLIT && nufft_tiles(p->n_virt, C, r->n_samples, p->path_cap) &&
        w.Qg >= w.Qn * std::min(C, kTile)) {
      launch_chirps(p, r, w, cube, st);
      return SBR_OK;
    }
    const int wave = std::min(w.Qg, nufft_wave(p->n_virt, w.Qn, C, r->n_samples));
    int best = 1, group = 1;
    double cost = 1e30;
    for (int q = 1; q <= w.Qn; ++q) {
      const int most = std::min(w.rows, wave / q), launches = (C + most - 1) / most;
      if (launches < cost * q) {
        cost = (double)launches / q;
        best = q;
        group = (C + launches - 1) / launches;
      }
    }
    for (int c = 0; c < C; c += group)
      launch_nufft(mode, p, r, w, true, best, c, std::min(group, C - c), cube, st);
    return SBR_OK;
  }
  set_error("sbr_synthesize: SBR_SYNTH_MOVING supports SBR_PHASE_SPLIT up to %d samples and SBR_PHASE_FP64",
            kNuMovingMaxSamples);
  return SBR_ERR_UNSUPPORTED;
}

template <int M>
void launch_fwd(sbr_phase_mode mode, const sbr_paths* p, const sbr_radar_cfg* r, const SynthWs& w,
                cudaStream_t st) {
  const int V = p->n_virt, Ns = r->n_samples, T = Ns / M;
  const int grid = V * w.Q;
  const float4* prep = reinterpret_cast<const float4*>(p->prep);
  if (mode == SBR_PHASE_SPLIT && (Ns == 256 || Ns == 512)) {
    ::sbr::note_launch();
    if (Ns == 256) launch_after(k_synth_mma<1>, grid, kMmaThreads, 0, st, prep, p->path_cap, p->count, V, w.Q,
                                w.partial);
    else launch_after(k_synth_mma<2>, grid, kMmaThreads, 0, st, prep, p->path_cap, p->count, V, w.Q, w.partial);
  } else if (mode == SBR_PHASE_SPLIT) {
    ::sbr::note_launch();
    launch_after(k_synth_split<M>, grid, kSplitThreads, split_smem(Ns), st, prep, p->path_cap, p->count, V, w.Q, Ns,
                 w.partial);
  } else if (mode == SBR_PHASE_FP64) {
    ::sbr::note_launch();
    launch_after(k_synth_fp64<M>, grid, T, 0, st, prep, reinterpret_cast<const float2*>(p->path_len), p->phase_ofs,
                 p->path_cap, p->count, V, w.Q, Ns, r->f0, r->bandwidth / Ns, w.partial);
  } else {
    const double mu = r->bandwidth / r->chirp_time, dt = r->chirp_time / Ns;
    const float2* plen = reinterpret_cast<const float2*>(p->path_len);
    const float f0 = (float)r->f0, fmu = (float)mu, fdt = (float)dt;
    ::sbr::note_launch();
    // Several of its small CTAs to an SM: placed while the kernel before still holds some SMs,
    // they crowd the others for the whole launch (4 antennas x 800,000 records x 1024 samples
    // 2.23 ms launched after it, 2.94 dispatched early; 12 x 150,000 x 256 0.89 and 1.14).
    if (grid > sm_count())
      k_synth_naive<M><<<grid, T, 0, st>>>(prep, plen, p->phase_ofs, p->path_cap, p->count, V, w.Q, Ns, f0, fmu, fdt,
                                           w.partial);
    else
      launch_after(k_synth_naive<M>, grid, T, 0, st, prep, plen, p->phase_ofs, p->path_cap, p->count, V, w.Q, Ns, f0,
                   fmu, fdt, w.partial);
  }
}
}  // namespace

extern "C" sbr_status sbr_synthesize(const sbr_paths* paths, const sbr_radar_cfg* radar,
                                     sbr_phase_mode mode_flags, float* d_cube, void* d_ws,
                                     size_t ws_bytes, sbr_stream stream) {
  SBR_ARG(paths && d_cube, "sbr_synthesize: NULL paths or cube");
  const bool moving = ((int)mode_flags & SBR_SYNTH_MOVING) != 0;
  const sbr_phase_mode mode = (sbr_phase_mode)((int)mode_flags & ~SBR_SYNTH_MOVING);
  sbr_status rs = check_radar(radar, "sbr_synthesize");
  if (rs != SBR_OK) return rs;
  SBR_ARG(paths->n_virt == radar->n_tx * radar->n_rx, "sbr_synthesize: paths have V=%d, radar %d",
          paths->n_virt, radar->n_tx * radar->n_rx);
  SBR_ARG(mode == SBR_PHASE_SPLIT || mode == SBR_PHASE_FP64 || mode == SBR_PHASE_NAIVE,
          "sbr_synthesize: unknown phase mode %d", (int)mode);
  SynthWs w;
  rs = bind_ws(radar, paths->path_cap, moving, d_ws, ws_bytes, &w, "sbr_synthesize");
  if (rs != SBR_OK) return rs;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int Ns = radar->n_samples, T = threads_for(Ns), M = Ns / T;
  if (moving) {
    rs = launch_moving(mode, paths, radar, w, reinterpret_cast<float2*>(d_cube), st);
    if (rs != SBR_OK) return rs;
    SBR_CUDA(cudaGetLastError());
    return SBR_OK;
  }
  if (nufft_for(mode, Ns, paths->path_cap * paths->n_virt)) {
    launch_nufft(mode, paths, radar, w, false, w.Qn, 0, 1, reinterpret_cast<float2*>(d_cube), st);
    SBR_CUDA(cudaGetLastError());
    return SBR_OK;
  }
  switch (M) {
    case 1: launch_fwd<1>(mode, paths, radar, w, st); break;
    case 2: launch_fwd<2>(mode, paths, radar, w, st); break;
    case 4: launch_fwd<4>(mode, paths, radar, w, st); break;
    case 8: launch_fwd<8>(mode, paths, radar, w, st); break;
    case 16: launch_fwd<16>(mode, paths, radar, w, st); break;
    default: set_error("sbr_synthesize: no kernel for %d samples per thread", M); return SBR_ERR_UNSUPPORTED;
  }
  SBR_CUDA(cudaGetLastError());
  const int V = paths->n_virt;
  ::sbr::note_launch();
  launch_after(k_reduce, reduce_grid(V, Ns, radar->n_chirps), 256, 0, st, w.partial, V, w.Q, Ns, radar->n_chirps,
               reinterpret_cast<float2*>(d_cube));
  SBR_CUDA(cudaGetLastError());
  return SBR_OK;
}

// ---- allocation-free variant ------------------------------------------------
//
// For callers that cannot call cudaMalloc (or reserve any device memory of
// their own) at the point where they synthesise: hosts that hand out no device
// allocator to plugins, real-time loops that must not risk the implicit device
// synchronisation of an allocation, or code running under a frozen memory
// budget.  The per-CTA partial sums then live in a fixed file-scope device
// array instead of a caller workspace.

namespace {
constexpr size_t kStaticPartials = 131072;  // float2 entries: 1 MiB on every device using the library
__device__ __align__(256) float2 g_static_partials[kStaticPartials];

constexpr int kMaxDevices = 64;
float2* g_static_ptr[kMaxDevices] = {};
std::mutex g_static_mu;

// Device address of the array for the current device (host code only holds a
// stand-in symbol).  Looked up once per device, on that device's first call.
sbr_status static_partials(float2** out) {
  int dev = -1;
  SBR_CUDA(cudaGetDevice(&dev));
  SBR_ARG(dev >= 0 && dev < kMaxDevices, "sbr_synthesize_noalloc: device %d beyond %d", dev, kMaxDevices);
  std::lock_guard<std::mutex> lock(g_static_mu);
  if (!g_static_ptr[dev]) {
    void* p = nullptr;
    SBR_CUDA(cudaGetSymbolAddress(&p, g_static_partials));
    g_static_ptr[dev] = static_cast<float2*>(p);
  }
  *out = g_static_ptr[dev];
  return SBR_OK;
}
}  // namespace

extern "C" sbr_status sbr_synthesize_noalloc(const sbr_paths* paths, const sbr_radar_cfg* radar,
                                             sbr_phase_mode mode, float* d_cube, sbr_stream stream) {
  SBR_ARG(paths && d_cube, "sbr_synthesize_noalloc: NULL paths or cube");
  sbr_status rs = check_radar(radar, "sbr_synthesize_noalloc");
  if (rs != SBR_OK) return rs;
  SBR_ARG(paths->n_virt == radar->n_tx * radar->n_rx, "sbr_synthesize_noalloc: paths have V=%d, radar %d",
          paths->n_virt, radar->n_tx * radar->n_rx);
  SBR_ARG(mode == SBR_PHASE_SPLIT || mode == SBR_PHASE_FP64 || mode == SBR_PHASE_NAIVE,
          "sbr_synthesize_noalloc: unknown phase mode %d", (int)mode);
  const int V = paths->n_virt, Ns = radar->n_samples;
  const size_t row = (size_t)V * Ns;  // one partial cube (one CTA per antenna)
  if (row > kStaticPartials) {
    set_error("sbr_synthesize_noalloc: V * N_s = %zu partial sums exceed the fixed scratch of %zu "
              "(1 MiB); use sbr_synthesize with a workspace",
              row, kStaticPartials);
    return SBR_ERR_UNSUPPORTED;
  }
  SynthWs w;
  rs = static_partials(&w.partial);
  if (rs != SBR_OK) return rs;
  w.gsum = nullptr;
  grid_shape(V, Ns, paths->path_cap, &w.Q);
  const int qmax = (int)(kStaticPartials / row);
  if (w.Q > qmax) w.Q = qmax;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int T = threads_for(Ns), M = Ns / T;
  switch (M) {
    case 1: launch_fwd<1>(mode, paths, radar, w, st); break;
    case 2: launch_fwd<2>(mode, paths, radar, w, st); break;
    case 4: launch_fwd<4>(mode, paths, radar, w, st); break;
    case 8: launch_fwd<8>(mode, paths, radar, w, st); break;
    case 16: launch_fwd<16>(mode, paths, radar, w, st); break;
    default: set_error("sbr_synthesize_noalloc: no kernel for %d samples per thread", M); return SBR_ERR_UNSUPPORTED;
  }
  SBR_CUDA(cudaGetLastError());
  ::sbr::note_launch();
  launch_after(k_reduce, reduce_grid(V, Ns, radar->n_chirps), 256, 0, st, w.partial, V, w.Q, Ns, radar->n_chirps,
               reinterpret_cast<float2*>(d_cube));
  SBR_CUDA(cudaGetLastError());
  return SBR_OK;
}

extern "C" sbr_status sbr_synthesize_bwd(const sbr_paths* paths, const sbr_radar_cfg* radar,
                                         const float* d_gcube, float* d_glen, float* d_gamp, float* d_gphase,
                                         void* d_ws, size_t ws_bytes, sbr_stream stream) {
  SBR_ARG(paths && d_gcube && d_glen && d_gamp, "sbr_synthesize_bwd: NULL argument");
  sbr_status rs = check_radar(radar, "sbr_synthesize_bwd");
  if (rs != SBR_OK) return rs;
  SBR_ARG(paths->n_virt == radar->n_tx * radar->n_rx, "sbr_synthesize_bwd: V mismatch");
  SynthWs w;
  rs = bind_ws(radar, paths->path_cap, false, d_ws, ws_bytes, &w, "sbr_synthesize_bwd");
  if (rs != SBR_OK) return rs;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int V = paths->n_virt, Ns = radar->n_samples, C = radar->n_chirps;
  const double lam_inv = radar->f0 / kC;
  if (paths->path_cap > 0 && adj_nufft_for(Ns, C, paths->path_cap * V)) {
    int log_m = 0;
    while ((1 << log_m) < 2 * Ns) ++log_m;
    SBR_CUDA(adj_attr(Ns));
    cudaLaunchConfig_t lc{};
    cudaLaunchAttribute at[2] = {};
    const unsigned ranks = C >= 8 ? 8 : 2;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = ranks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // as launch_after
    at[1].val.programmaticStreamSerializationAllowed = 1;
    lc.gridDim = dim3(V * ranks);
    lc.blockDim = dim3(kAdjThreads);
    lc.dynamicSmemBytes = adj_smem(Ns);
    lc.stream = st;
    lc.attrs = at;
    lc.numAttrs = 2;
    const NufftCoef& co = nufft_coef();
    ::sbr::note_launch();
    SBR_CUDA(cudaLaunchKernelEx(&lc, k_adj_grid, reinterpret_cast<const float2*>(d_gcube), V, C, Ns, log_m,
                                (float)(radar->bandwidth / (radar->f0 * Ns)), co, reinterpret_cast<float2*>(w.adj)));
    // a wave of CTAs at most, at least one per antenna
    const int64_t need = (paths->path_cap + 255) / 256, wave = std::max(1, 8 * sm_count() / V);
    ::sbr::note_launch();
    launch_after(k_synth_bwd_nufft, dim3((unsigned)std::min(need, wave), V), 256, 0, st,
                 reinterpret_cast<const float4*>(paths->prep), paths->path_cap, paths->count, log_m, co, w.adj,
                 (float)lam_inv, d_glen, d_gamp, d_gphase);
    SBR_CUDA(cudaGetLastError());
    return SBR_OK;
  }
  // the upstream gradient summed over the (equal) chirps; one chirp needs no sum
  const float2* gs = reinterpret_cast<const float2*>(d_gcube);
  if (C > 1) {
    ::sbr::note_launch();
    launch_after(k_chirp_sum, (V * Ns + 255) / 256, 256, 0, st, gs, V, C, Ns, w.gsum);
    gs = w.gsum;
  }
  const int64_t cap = paths->path_cap;
  if (cap > 0) {
    dim3 grid((unsigned)((cap + 255) / 256), (unsigned)V);
    const double bcn = radar->bandwidth / (kC * Ns);
    ::sbr::note_launch();
    launch_after(k_synth_bwd, grid, 256, Ns * sizeof(float2), st, reinterpret_cast<const float4*>(paths->prep), cap,
                 paths->count, Ns, gs, (float)lam_inv, (float)bcn, d_glen, d_gamp, d_gphase);
  }
  SBR_CUDA(cudaGetLastError());
  return SBR_OK;
}
