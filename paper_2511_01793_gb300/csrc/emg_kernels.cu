// Kernels of the eMAGPIE hot path (arXiv 2511.01793) for sm_103a.
//
//   k_amp_prep     a_k = sqrt(max(d_k, 0)) reordered into the FFT storage order
//   k_prep         per-minibatch probe-only arrays: max|Q|^2, gains G_l, MAGPIE
//                  weights W_z, W_R and restricted probes Q_l (Sec. 3.2)
//   k_stepc<M, C>  one cluster of C CTAs per scan position: gather, exit wave, 2-D FFT,
//                  modulus replacement (Def. 2.1), inverse FFT, MAGPIE object step,
//                  ePIE probe step, geometric-mean joint step (Eq. geomean)
//   k_step<M>      the same in one CTA, for the allocation-free entry point
//   k_apply        deterministic combine of the minibatch into object and probe
//   k_forward<M>   Phi_k = 1/2 ||Q . P_k z - R_k||^2 (Eq. exit_misfit) per position,
//                  d_k = |F(Q . P_k z)|^2 (Sec. 2.1 data model), batched 2-D DFT
//                  of natural-order tiles
#include <cooperative_groups.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <type_traits>

#include "emg_fft.cuh"
#include "emg_internal.h"

namespace emg {
namespace {
#ifdef EMG_BOUNDS_CHECK
__device__ unsigned g_bounds_error;
__device__ __forceinline__ bool in_bounds(long long i, long long n, int site) {
  if (i >= 0 && i < n) return true;
  atomicOr(&g_bounds_error, 1u << site);
  return false;
}
#define EMG_INB(i, n, site) in_bounds((long long)(i), (long long)(n), (site))
#else
#define EMG_INB(i, n, site) true
#endif
}  // namespace

#ifdef EMG_BOUNDS_CHECK
namespace {
// Exercises the recording path of the checks: index n against a bound of n
// fails the check, so the store is skipped (buf holds n + 1 floats regardless).
__global__ void k_bounds_probe(float* buf, int n) {
  if (threadIdx.x == 0 && EMG_INB(n, n, kBcLevel)) buf[n] = 1.f;
}
}  // namespace
#endif

cudaError_t bounds_probe(unsigned* out) {
#ifdef EMG_BOUNDS_CHECK
  float* buf = nullptr;
  const int n = 32;
  cudaError_t e = cudaMalloc(&buf, (n + 1) * sizeof(float));
  if (e != cudaSuccess) return e;
  k_bounds_probe<<<1, 32>>>(buf, n);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  cudaFree(buf);
  if (e != cudaSuccess) return e;
  return bounds_errors_take(out);
#else
  *out = 0;
  return cudaErrorNotSupported;
#endif
}

cudaError_t bounds_errors_take(unsigned* out) {
#ifdef EMG_BOUNDS_CHECK
  unsigned zero = 0;
  cudaError_t e = cudaMemcpyFromSymbol(out, g_bounds_error, sizeof(unsigned));
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_bounds_error, &zero, sizeof(unsigned));
  return e;
#else
  *out = 0;
  return cudaErrorNotSupported;
#endif
}
}  // namespace emg

namespace emg {

namespace {

template <int M> struct StepThreads;
template <> struct StepThreads<16> { static constexpr int value = 64; };
template <> struct StepThreads<32> { static constexpr int value = 128; };
template <> struct StepThreads<64> { static constexpr int value = 256; };
template <> struct StepThreads<128> { static constexpr int value = 512; };

__device__ __forceinline__ float2 czero() { return make_float2(0.f, 0.f); }

// Programmatic dependent launch: the minibatch kernels (prep -> step ->
// combine) are launched so that each may start while its predecessor drains.
// pdl_wait() blocks until the predecessor grid has finished and its writes are
// visible; everything before it may only read data that no predecessor
// writes (scan order, positions, amplitudes).  pdl_trigger() lets the
// successor launch.  Both are no-ops for an ordinary launch.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Cluster barrier arrive without release semantics, for barriers that order
// execution only (every CTA of the cluster resident; no CTA exits while a
// neighbour still reads its shared memory).  A release arrive would first
// wait for all of the thread's outstanding loads and stores.
__device__ __forceinline__ void cluster_arrive_relaxed() {
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.aligned;" ::: "memory"); }

// 16-byte asynchronous copies into shared memory (both addresses 16-byte aligned).
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ float2 gather_obj(const float2* __restrict__ z, int n_rows, int n_cols,
                                             int gr, int gc) {
  if ((unsigned)gr < (unsigned)n_rows && (unsigned)gc < (unsigned)n_cols)
    return z[(size_t)gr * n_cols + gc];
  return czero();
}

// num / den with 0/0 read as 0 (den == 0 gives 0).
__device__ __forceinline__ float safe_div(float num, float den) { return den != 0.f ? num / den : 0.f; }
__device__ __forceinline__ float2 safe_cdiv(float2 num, float den) {
  return den != 0.f ? make_float2(num.x / den, num.y / den) : czero();
}

// Principal square root of w (Kahan, "Branch cuts for complex elementary functions", 1987).
__device__ __forceinline__ float2 csqrt_principal(float2 w) {
  const float mag = sqrtf(fmaf(w.x, w.x, w.y * w.y));
  if (mag == 0.f) return czero();
  const float t = sqrtf(0.5f * (fabsf(w.x) + mag));
  if (w.x >= 0.f) return make_float2(t, w.y / (2.f * t));
  return make_float2(fabsf(w.y) / (2.f * t), copysignf(t, w.y));
}

// y with y^2 = x * xp and Re(y conj(x)) >= 0 (Eq. geomean); ties keep the principal root.
__device__ __forceinline__ float2 geometric_mean_aligned(float2 x, float2 xp) {
  float2 y = csqrt_principal(cmul(x, xp));
  if (fmaf(y.x, x.x, y.y * x.y) < 0.f) y = make_float2(-y.x, -y.y);
  return y;
}

// c + a b, c - a b and c + conj(a) b as chains of two fused multiply-adds per part.
__device__ __forceinline__ float2 cfma(float2 a, float2 b, float2 c) {
  return make_float2(fmaf(a.x, b.x, fmaf(-a.y, b.y, c.x)), fmaf(a.x, b.y, fmaf(a.y, b.x, c.y)));
}
__device__ __forceinline__ float2 cfnma(float2 a, float2 b, float2 c) {
  return make_float2(fmaf(-a.x, b.x, fmaf(a.y, b.y, c.x)), fmaf(-a.x, b.y, fmaf(-a.y, b.x, c.y)));
}
__device__ __forceinline__ float2 cfma_conj(float2 a, float2 b, float2 c) {
  return make_float2(fmaf(a.x, b.x, fmaf(a.y, b.y, c.x)), fmaf(a.x, b.y, fmaf(-a.y, b.x, c.y)));
}

// y with y^2 = x * xp and Re(y conj(x)) >= 0 (Eq. geomean), branch-free.
// With w = x xp = u + i v, s = (|u| + |w|)/2, t = sqrt(s), h = 1/(2t): (t, v h)
// squares to w when u >= 0 (Kahan's half-angle form), and (v h, t) when u < 0
// (its real part is (v^2 - 4 s^2)/(4 s) = u).  With s' = 2 s and r = 1 / sqrt(s'),
// t = s' r / sqrt(2) and v h = v r / sqrt(2).
// A floor of 1e-37 under both square roots gives y = 0 for w = 0 without a
// branch; it changes no result for |w|^2 above about 1e-29.  The sign flip
// is applied to the sign bit when Re(y conj(x)) < 0.
__device__ __forceinline__ float2 geomean_aligned_root(float2 x, float2 xp) {
  const float2 w = cmul(x, xp);
  const float n = fmaf(w.x, w.x, w.y * w.y);
  const float mag = n * rsqrtf(n + 1e-37f);
  const float s2 = fabsf(w.x) + mag;
  const float rr = rsqrtf(s2 + 1e-37f) * 0.70710678118654752f;
  const float t = s2 * rr, vh = w.y * rr;
  const float yx = w.x >= 0.f ? t : vh, yy = w.x >= 0.f ? vh : t;
  const unsigned sbit = fmaf(yx, x.x, yy * x.y) < 0.f ? 0x80000000u : 0u;
  return make_float2(__uint_as_float(__float_as_uint(yx) ^ sbit), __uint_as_float(__float_as_uint(yy) ^ sbit));
}

// geometric_mean_aligned without its branches and the slow paths of IEEE roots and division: from the
// rsqrt unit, with one Newton step each for |w|, t and v h, which leaves about the rounding of correctly
// rounded operations.  Where |w|^2 is an FP32 number at all the lower bounds under the roots change
// nothing (s >= |w| / 2 >= 5.4e-20), so there is no floor; w = 0 gives 0, a tie keeps the principal root.
__device__ __forceinline__ float2 geometric_mean_rounded(float2 x, float2 xp) {
  const float2 w = cmul(x, xp);
  const float n = fmaf(w.x, w.x, w.y * w.y);
  const float r = rsqrtf(fmaxf(n, 1.17549435e-38f));
  float mag = n * r;
  mag = fmaf(0.5f * mag, fmaf(-mag, r, 1.f), mag);  // the residual of r, of size 1: it never underflows
  const float s = 0.5f * (fabsf(w.x) + mag);
  const float q = rsqrtf(fmaxf(s, 5e-20f)), h = 0.5f * q;  // h = 1 / (2 t)
  float t = s * q;
  t = fmaf(fmaf(-t, t, s), h, t);
  float vh = w.y * h;
  vh = fmaf(fmaf(-2.f * t, vh, w.y), h, vh);
  const unsigned sv = w.x < 0.f ? __float_as_uint(w.y) & 0x80000000u : 0u;  // (|v h|, t sign(v)) when u < 0
  const float yx = w.x < 0.f ? vh : t, yy = w.x < 0.f ? t : vh;
  const float2 y = make_float2(__uint_as_float(__float_as_uint(yx) ^ sv), __uint_as_float(__float_as_uint(yy) ^ sv));
  const unsigned sbit = fmaf(y.x, x.x, y.y * x.y) < 0.f ? 0x80000000u : 0u;
  return make_float2(__uint_as_float(__float_as_uint(y.x) ^ sbit), __uint_as_float(__float_as_uint(y.y) ^ sbit));
}

// a5 (finest level) + a6 + a7 at one pixel: with MG the fine MAGPIE step from
// the prolonged coarse correction pro, z^+ = zp + G_0 (R - Q zp) with
// zp = z_k + pro, else z^+ = z_k + G_0 (R - Q z_k); Q^+ = Q + conj(z_k)(R - Q z_k)/mu_k;
// with JOINT their aligned geometric means with z_k and Q (Eq. geomean), to the
// accuracy of correctly rounded roots (ROUNDED) or of the rsqrt unit.
template <bool MG, bool JOINT, bool ROUNDED>
__device__ __forceinline__ void update_pixel(float2 zk, float2 q, float2 g0, float2 R, float2 pro, float inv_mu,
                                             float2& zn, float2& qn) {
  const float2 res = cfnma(q, zk, R);
  float2 zplus;
  if constexpr (MG) {
    const float2 zp = cadd(zk, pro);
    zplus = cfma(g0, cfnma(q, zp, R), zp);
  } else {
    zplus = cfma(g0, res, zk);
  }
  const float2 qplus = cfma_conj(zk, cscale(res, inv_mu), q);
  if constexpr (JOINT && ROUNDED) {
    zn = geometric_mean_rounded(zk, zplus);
    qn = geometric_mean_rounded(q, qplus);
  } else if constexpr (JOINT) {
    zn = geomean_aligned_root(zk, zplus);
    qn = geomean_aligned_root(q, qplus);
  } else {
    zn = zplus;
    qn = qplus;
  }
}

// Atomic object scatter of one patch pixel (EMG_SCATTER_ATOMIC): weighted mean
// (combine 0) adds w z~ and w, the summed corrections (combine 1) add z~ - z_k.
__device__ __forceinline__ void scatter_atomic(float2* num, float* den, int combine, int n_rows, int n_cols, int gr,
                                               int gc, float2 zn, float2 zk, float w) {
  if ((unsigned)gr >= (unsigned)n_rows || (unsigned)gc >= (unsigned)n_cols) return;
  const size_t gi = (size_t)gr * n_cols + gc;
  if (combine == 0) {
    atomicAdd(num + gi, make_float2(w * zn.x, w * zn.y));
    atomicAdd(den + gi, w);
  } else {
    atomicAdd(num + gi, make_float2(zn.x - zk.x, zn.y - zk.y));
  }
}

template <typename T>
__device__ __forceinline__ T lerp4(T a, T b, T c, T d);
template <>
__device__ __forceinline__ float lerp4<float>(float a, float b, float c, float d) {
  return 0.5625f * a + 0.1875f * b + 0.1875f * c + 0.0625f * d;
}
template <>
__device__ __forceinline__ float2 lerp4<float2>(float2 a, float2 b, float2 c, float2 d) {
  return make_float2(lerp4<float>(a.x, b.x, c.x, d.x), lerp4<float>(a.y, b.y, c.y, d.y));
}

// (I_H^h y)(r, c) for a coarse array of side mc with row stride `stride`.
// kind 0: piecewise constant (4 (I_h^H)^T); kind 1: cell-centred bilinear, edge clamp.
template <typename T>
__device__ __forceinline__ T prolong_at(const T* y, int stride, int mc, int r, int c, int kind) {
  const int i = r >> 1, j = c >> 1;
  const T v = y[i * stride + j];
  if (kind == 0) return v;
  const int i2 = (r & 1) ? min(i + 1, mc - 1) : max(i - 1, 0);
  const int j2 = (c & 1) ? min(j + 1, mc - 1) : max(j - 1, 0);
  return lerp4<T>(v, y[i2 * stride + j], y[i * stride + j2], y[i2 * stride + j2]);
}

template <int NT>
__device__ __forceinline__ float block_max(float v, float* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = sh[0];
#pragma unroll
  for (int i = 1; i < NT / 32; ++i) r = fmaxf(r, sh[i]);
  __syncthreads();
  return r;
}

// Sum over the block of per-thread FP32 partials: FP32 warp trees, then the
// NT/32 warp sums added in FP64 by one thread in a fixed order; the result is
// broadcast.  Deterministic; avoids FP64 work in every thread.
template <int NT>
__device__ __forceinline__ double block_sum_f(float v, float* shf, double* shd) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) shf[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double r = 0.0;
#pragma unroll
    for (int i = 0; i < NT / 32; ++i) r += (double)shf[i];
    shd[0] = r;
  }
  __syncthreads();
  return shd[0];
}

// FP64 block sum, broadcast: warp trees, then one warp's tree over the NT/32
// warp sums.  (The FP64 pipe takes two results per SM and clock: every thread
// adding all warp sums cost 8 us in a block of 1024.)
template <int NT>
__device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    double r = threadIdx.x < NT / 32 ? sh[threadIdx.x] : 0.0;
#pragma unroll
    for (int o = NT / 64; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    if (threadIdx.x == 0) sh[0] = r;
  }
  __syncthreads();
  const double r = sh[0];
  __syncthreads();
  return r;
}

// Warp sum of FP32 values without the FP64 pipe, to about 48 bits: each tree
// level adds exactly (Knuth's TwoSum) and carries the rounding errors along.
// Every lane has the same `hi`, so where the sum leaves the FP32 range (or a value
// is not finite) the whole warp adds in FP64.  Lane 0 gets the value.
__device__ __forceinline__ double warp_sum_exact(float v) {
  float hi = v, lo = 0.f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float b = __shfl_xor_sync(0xffffffffu, hi, o), bl = __shfl_xor_sync(0xffffffffu, lo, o);
    const float s = hi + b, t = s - hi;
    lo += bl + ((hi - (s - t)) + (b - t));
    hi = s;
  }
  if (isfinite(hi)) return (double)hi + (double)lo;
  double s = v;
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// ---------------------------------------------------------------------------
// a_k in storage order: amp[k][e_r][e_c] = sqrt(max(d[k][f(e_r)][f(e_c)], 0)).
// Warp-level max (sum) of v, written by lane 0 of each warp to sh[warp]; after
// a barrier, partials_max / partials_sum combine them in warp order (the sums in
// FP64), so a caller can let one existing barrier serve.
__device__ __forceinline__ void warp_partial_max(float v, float* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
}
template <typename V>
__device__ __forceinline__ void warp_partial_sum(V v, V* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
}
template <int NT>
__device__ __forceinline__ float partials_max(const float* sh) {
  float r = sh[0];
#pragma unroll
  for (int i = 1; i < NT / 32; ++i) r = fmaxf(r, sh[i]);
  return r;
}
template <int NT, typename V>
__device__ __forceinline__ double partials_sum(const V* sh) {
  double r = 0.0;
#pragma unroll
  for (int i = 0; i < NT / 32; ++i) r += (double)sh[i];
  return r;
}

template <int M>
__global__ void __launch_bounds__(256) k_amp_prep(const float* __restrict__ d, float* __restrict__ amp,
                                                  int n_pos) {
  // One warp per storage row: the frequency row it needs is read whole with
  // consecutive lanes on consecutive words (the source may be host memory read
  // over the CPU-GPU link), then permuted through shared memory.
  constexpr int PL = (M + 31) / 32;
  __shared__ float rows[8][M];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* buf = rows[warp];
  const size_t n_rows = (size_t)n_pos * M;
  for (size_t g = (size_t)blockIdx.x * 8 + warp; g < n_rows; g += (size_t)gridDim.x * 8) {
    const size_t k = g / M;
    const int er = (int)(g % M);
    const float* src = d + (k * M + storage_to_freq<M>(er)) * M;
    float v[PL];
#pragma unroll
    for (int j = 0; j < PL; ++j)
      if (lane + 32 * j < M) v[j] = src[lane + 32 * j];
#pragma unroll
    for (int j = 0; j < PL; ++j)
      if (lane + 32 * j < M) buf[lane + 32 * j] = v[j];
    __syncwarp();
    float* dst = amp + g * M;
#pragma unroll
    for (int j = 0; j < PL; ++j) {
      const int ec = lane + 32 * j;
      if (ec < M) dst[ec] = sqrtf(fmaxf(buf[storage_to_freq<M>(ec)], 0.f));
    }
    __syncwarp();
  }
}

// a_k of the positions idx[0..b) into their slots of amp, read from d (any
// device-readable address, e.g. pinned host memory).  A small grid that runs
// beside the step kernels: each warp keeps kGatherRows rows of loads in flight.
#ifndef EMG_GATHER_BLOCKS
#define EMG_GATHER_BLOCKS 38
#endif
#ifndef EMG_GATHER_ROWS
#define EMG_GATHER_ROWS 4
#endif
#ifndef EMG_GATHER_WARPS
#define EMG_GATHER_WARPS 8
#endif
constexpr int kGatherRows = EMG_GATHER_ROWS, kGatherWarps = EMG_GATHER_WARPS, kGatherBlocks = EMG_GATHER_BLOCKS;
template <int M>
__global__ void __launch_bounds__(kGatherWarps * 32) k_amp_gather(const float* __restrict__ d,
                                                                 const int32_t* __restrict__ idx, int b,
                                                                 float* __restrict__ amp) {
  constexpr int PL = (M + 31) / 32, RW = kGatherRows;
  static_assert(M % RW == 0, "row groups stay within one position");
  __shared__ __align__(16) float rows[kGatherWarps][RW][M];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_groups = b * (M / RW);
  // rows of M >= 128 floats at a 16-byte aligned source: one 16-byte load per
  // lane and 128 columns, fewer and larger reads over the CPU-GPU link
  constexpr int PV = M / 128;
  const bool vec = PV > 0 && (reinterpret_cast<uintptr_t>(d) & 15) == 0;
  for (int g = blockIdx.x * kGatherWarps + warp; g < n_groups; g += gridDim.x * kGatherWarps) {
    const int kk = g / (M / RW), er0 = (g % (M / RW)) * RW;
    const size_t k = (size_t)idx[kk];
    if constexpr (PV > 0) {
      if (vec) {
        float4 v4[RW][PV];
#pragma unroll
        for (int r = 0; r < RW; ++r) {
          const float4* src = reinterpret_cast<const float4*>(d + (k * M + storage_to_freq<M>(er0 + r)) * M);
#pragma unroll
          for (int j = 0; j < PV; ++j) v4[r][j] = src[lane + 32 * j];
        }
#pragma unroll
        for (int r = 0; r < RW; ++r)
#pragma unroll
          for (int j = 0; j < PV; ++j) *reinterpret_cast<float4*>(&rows[warp][r][4 * (lane + 32 * j)]) = v4[r][j];
      }
    }
    if (!vec) {
      float v[RW][PL];
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        const float* src = d + (k * M + storage_to_freq<M>(er0 + r)) * M;
#pragma unroll
        for (int j = 0; j < PL; ++j)
          if (lane + 32 * j < M) v[r][j] = src[lane + 32 * j];
      }
#pragma unroll
      for (int r = 0; r < RW; ++r)
#pragma unroll
        for (int j = 0; j < PL; ++j)
          if (lane + 32 * j < M) rows[warp][r][lane + 32 * j] = v[r][j];
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      float* dst = amp + (k * M + er0 + r) * M;
#pragma unroll
      for (int j = 0; j < PL; ++j) {
        const int ec = lane + 32 * j;
        if (ec < M) dst[ec] = sqrtf(fmaxf(rows[warp][r][storage_to_freq<M>(ec)], 0.f));
      }
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// Probe-only arrays of one minibatch (single CTA; O(m^2) work).
constexpr int kPrepThreads = 1024;

__global__ void __launch_bounds__(kPrepThreads) k_prep(const PrepArgs a) {
  __shared__ float redf[kPrepThreads / 32];
  const int tid = threadIdx.x;
  const int m = a.m;
  float mx = 0.f;
  for (int p = tid; p < m * m; p += kPrepThreads) mx = fmaxf(mx, cabs2(a.probe[p]));
  const float MQ = block_max<kPrepThreads>(mx, redf);
  if (tid == 0 && a.mq_next) *a.mq_next = 0u;

  // level 0: u_0 = alpha (M_Q - |Q|^2), G_0, combine weight
  for (int p = tid; p < m * m; p += kPrepThreads) {
    const float2 q = a.probe[p];
    const float a2 = cabs2(q);
    const float u = a.alpha * (MQ - a2);
    a.u[0][p] = u;
    a.G[0][p] = safe_cdiv(cconj(q), u + a2);
    a.wq[p] = fmaf(a.w_eps, MQ, a2);
  }
  for (int l = 0; l + 1 < a.levels; ++l) {
    __syncthreads();
    const int mf = m >> l, mc = mf >> 1;
    const float2* Qf = (l == 0) ? a.probe : a.Q[l];
    const float* uf = a.u[l];
    // coarse: T = I_h^H |Q_l|^2, Q_{l+1} = I_h^H Q_l, u_{l+1} = W_u^H I_h^H u_l, G_{l+1}
    for (int pc = tid; pc < mc * mc; pc += kPrepThreads) {
      const int i = pc / mc, j = pc % mc;
      float t = 0.f, ur = 0.f;
      float2 qs = czero();
#pragma unroll
      for (int dy = 0; dy < 2; ++dy)
#pragma unroll
        for (int dx = 0; dx < 2; ++dx) {
          const int pf = (2 * i + dy) * mf + 2 * j + dx;
          const float2 q = Qf[pf];
          t += cabs2(q);
          qs = cadd(qs, q);
          ur += uf[pf];
        }
      t *= 0.25f;
      ur *= 0.25f;
      qs = cscale(qs, 0.25f);
      const float aH = cabs2(qs);
      const float uH = safe_div(aH, t) * ur;
      a.T[l][pc] = t;
      a.Q[l + 1][pc] = qs;
      a.u[l + 1][pc] = uH;
      a.G[l + 1][pc] = safe_cdiv(cconj(qs), uH + aH);
    }
    __syncthreads();
    // fine: W_z = |Q_l|^2 / S, W_R = (I_H^h Q_{l+1}) conj(Q_l) / S, S = I_H^h T
    for (int pf = tid; pf < mf * mf; pf += kPrepThreads) {
      const int r = pf / mf, c = pf % mf;
      const float S = prolong_at<float>(a.T[l], mc, mc, r, c, a.prolong);
      const float2 pq = prolong_at<float2>(a.Q[l + 1], mc, mc, r, c, a.prolong);
      const float2 q = Qf[pf];
      a.Wz[l][pf] = safe_div(cabs2(q), S);
      a.WR[l][pf] = safe_cdiv(cmulc(pq, q), S);
    }
  }
}

// max|Q|^2 into *slot (float bits, atomicMax; the slot starts at 0).
__device__ __forceinline__ void warp_atomic_max(unsigned* slot, float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) atomicMax(slot, __float_as_uint(v));
}

// What precedes a call's first minibatch, in one launch: max|Q|^2 of the probe
// into mq[0], mq[1] and the ticket counters cleared, and (NI > 0) the
// minibatch's position indices, which travel in the launch parameters (the
// runtime copies them when the launch is enqueued, so the caller may overwrite
// its host array, pinned or not, once the call returns).  One cluster, so that
// the maximum needs no memory cleared beforehand.
constexpr int kSeedThreads = 512, kSeedCtas = 8, kSeedMaxIdx = 2048;
template <int NI>
struct SeedIdx {
  int32_t v[NI > 0 ? NI : 1];
};
template <int NI>
__global__ void __launch_bounds__(kSeedThreads) k_seed(const float2* __restrict__ probe, int n, unsigned* __restrict__ mq,
                                                       unsigned* __restrict__ sync, int32_t* __restrict__ order, int b,
                                                       const SeedIdx<NI> idx) {
  __shared__ float redf[kSeedThreads / 32];
  __shared__ float part[kSeedCtas];
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  const int rank = (int)cl.block_rank(), ctas = (int)cl.num_blocks(), tid = threadIdx.x;
  if (ctas > 1) cluster_arrive_relaxed();  // completed (wait) before the first distributed shared memory access
  pdl_wait();  // the probe and the counters belong to the previous kernel until it has ended
  float mx = 0.f;
#pragma unroll 8
  for (int p = rank * kSeedThreads + tid; p < n; p += ctas * kSeedThreads) mx = fmaxf(mx, cabs2(probe[p]));
  warp_partial_max(mx, redf);
  __syncthreads();
  if (ctas > 1) {
    cluster_wait();  // rank 0's CTA has started: its shared memory may be written
    if (tid == 0) *cl.map_shared_rank(&part[rank], 0) = partials_max<kSeedThreads>(redf);
    cl.sync();
  } else if (tid == 0) {
    part[0] = partials_max<kSeedThreads>(redf);
  }
  if (rank != 0) return;
  if (tid == 0) {
    float m = part[0];
    for (int d = 1; d < ctas; ++d) m = fmaxf(m, part[d]);
    mq[0] = __float_as_uint(m);
    mq[1] = 0u;
    if (sync) sync[0] = sync[1] = 0u;
  }
  if constexpr (NI > 0)
    for (int i = tid; i < b; i += kSeedThreads) order[i] = idx.v[i];
}

// Tiled probe-only prep: one CTA per tile x tile block of level-0 pixels.
// The CTA rebuilds the restriction pyramid of its tile plus a halo of
// 2^(L-1) px (bilinear prolongation reads one coarse neighbour per level) in
// shared memory and writes the level arrays of its own pixels.
constexpr int kPrepTileThreads = 256;

// Bounded wait of the fused prep: 1 s of %globaltimer, then the error flag.
constexpr unsigned long long kFusedPrepWaitNs = 1000000000ull;

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

struct PrepRegion {
  int lo_r, lo_c, h, w;   // region of one level, in that level's pixels
};

__device__ __forceinline__ PrepRegion prep_region(int m, int R0, int C0, int tile, int halo, int l) {
  PrepRegion g;
  const int lr = max(0, R0 - halo), hr = min(m, R0 + tile + halo);
  const int lc = max(0, C0 - halo), hc = min(m, C0 + tile + halo);
  g.lo_r = lr >> l;
  g.lo_c = lc >> l;
  g.h = (hr >> l) - g.lo_r;
  g.w = (hc >> l) - g.lo_c;
  return g;
}

// Prolongation at level-l pixel (r, c) from a coarse array stored on a region
// (row stride g.w, origin g.lo_r, g.lo_c); mc = full coarse side for clamping.
template <typename T>
__device__ __forceinline__ T prolong_region(const T* y, const PrepRegion& g, int mc, int r, int c, int kind) {
  const int i = r >> 1, j = c >> 1;
  const T v = y[(i - g.lo_r) * g.w + (j - g.lo_c)];
  if (kind == 0) return v;
  const int i2 = (r & 1) ? min(i + 1, mc - 1) : max(i - 1, 0);
  const int j2 = (c & 1) ? min(j + 1, mc - 1) : max(j - 1, 0);
  return lerp4<T>(v, y[(i2 - g.lo_r) * g.w + (j - g.lo_c)], y[(i - g.lo_r) * g.w + (j2 - g.lo_c)],
                  y[(i2 - g.lo_r) * g.w + (j2 - g.lo_c)]);
}

// The probe-only arrays of one tile (index `t`) of the probe, computed by
// `nt` threads of a CTA with `smp` as shared scratch (prep_tile_smem bytes).
__device__ __forceinline__ void prep_tile_body(const PrepArgs& a, int t, int tid, int nt, float2* smp) {
  const int m = a.m, L = a.levels, tile = a.tile, halo = a.halo;
  const int tiles_per_row = m / tile;
  const int R0 = (t / tiles_per_row) * tile, C0 = (t % tiles_per_row) * tile;
  const float MQ = __uint_as_float(*a.mq_read);
  if (t == 0 && tid == 0) *a.mq_next = 0u;

  // carve shared memory: per level Q_l (float2), u_l (float), T_l (float, level l+1 region)
  float2* Qs[kMaxLevels];
  float* us[kMaxLevels];
  float* Ts[kMaxLevels];
  {
    char* base = (char*)smp;
    size_t off = 0;
    for (int l = 0; l < L; ++l) {
      const PrepRegion g = prep_region(m, R0, C0, tile, halo, l);
      Qs[l] = (float2*)(base + off);
      off += (size_t)g.h * g.w * sizeof(float2);
      us[l] = (float*)(base + off);
      off += (size_t)g.h * g.w * sizeof(float);
      if (l + 1 < L) {
        const PrepRegion gc = prep_region(m, R0, C0, tile, halo, l + 1);
        Ts[l] = (float*)(base + off);
        off += (size_t)gc.h * gc.w * sizeof(float);
      }
      off = (off + 15) & ~(size_t)15;
    }
  }
  // level 0
  {
    const PrepRegion g = prep_region(m, R0, C0, tile, halo, 0);
    for (int p = tid; p < g.h * g.w; p += nt) {
      const int r = g.lo_r + p / g.w, c = g.lo_c + p % g.w;
      const float2 q = a.probe[r * m + c];
      const float a2 = cabs2(q);
      const float u = a.alpha * (MQ - a2);
      Qs[0][p] = q;
      us[0][p] = u;
      if (r >= R0 && r < R0 + tile && c >= C0 && c < C0 + tile) {
        a.G[0][r * m + c] = safe_cdiv(cconj(q), u + a2);
        a.wq[r * m + c] = fmaf(a.w_eps, MQ, a2);
      }
    }
  }
  for (int l = 0; l + 1 < L; ++l) {
    __syncthreads();
    const PrepRegion gf = prep_region(m, R0, C0, tile, halo, l);
    const PrepRegion gc = prep_region(m, R0, C0, tile, halo, l + 1);
    const int mf = m >> l, mc = mf >> 1;
    const int tr0 = R0 >> (l + 1), tc0 = C0 >> (l + 1), tsz = tile >> (l + 1);
    // coarse: T = I_h^H |Q_l|^2, Q_{l+1} = I_h^H Q_l, u_{l+1} = W_u^H I_h^H u_l, G_{l+1}
    for (int p = tid; p < gc.h * gc.w; p += nt) {
      const int i = p / gc.w, j = p % gc.w;
      float t = 0.f, ur = 0.f;
      float2 qs = czero();
#pragma unroll
      for (int dy = 0; dy < 2; ++dy)
#pragma unroll
        for (int dx = 0; dx < 2; ++dx) {
          const int pf = (2 * i + dy) * gf.w + 2 * j + dx;
          const float2 q = Qs[l][pf];
          t += cabs2(q);
          qs = cadd(qs, q);
          ur += us[l][pf];
        }
      t *= 0.25f;
      ur *= 0.25f;
      qs = cscale(qs, 0.25f);
      const float aH = cabs2(qs);
      const float uH = safe_div(aH, t) * ur;
      Ts[l][p] = t;
      Qs[l + 1][p] = qs;
      us[l + 1][p] = uH;
      const int gi = gc.lo_r + i, gj = gc.lo_c + j;
      if (gi >= tr0 && gi < tr0 + tsz && gj >= tc0 && gj < tc0 + tsz) {
        a.Q[l + 1][gi * mc + gj] = qs;
        a.G[l + 1][gi * mc + gj] = safe_cdiv(cconj(qs), uH + aH);
      }
    }
    __syncthreads();
    // fine weights of the tile's level-l pixels: W_z = |Q_l|^2 / S, W_R = (I_H^h Q_{l+1}) conj(Q_l) / S
    const int fr0 = R0 >> l, fc0 = C0 >> l, fsz = tile >> l;
    for (int p = tid; p < fsz * fsz; p += nt) {
      const int r = fr0 + p / fsz, c = fc0 + p % fsz;
      const float S = prolong_region<float>(Ts[l], gc, mc, r, c, a.prolong);
      const float2 pq = prolong_region<float2>(Qs[l + 1], gc, mc, r, c, a.prolong);
      const float2 q = Qs[l][(r - gf.lo_r) * gf.w + (c - gf.lo_c)];
      a.Wz[l][r * mf + c] = safe_div(cabs2(q), S);
      a.WR[l][r * mf + c] = safe_cdiv(cmulc(pq, q), S);
    }
  }
}

__global__ void __launch_bounds__(kPrepTileThreads) k_prep_tile(const PrepArgs a) {
  extern __shared__ float2 smp[];
  pdl_trigger();
  pdl_wait();  // the probe and max|Q|^2 come from the previous combine
  prep_tile_body(a, blockIdx.x, threadIdx.x, kPrepTileThreads, smp);
}

__host__ size_t prep_tile_smem(const PrepArgs& a) {
  // worst-case region sizes over tiles (interior tile)
  size_t bytes = 0;
  for (int l = 0; l < a.levels; ++l) {
    const int side = min(a.m, a.tile + 2 * a.halo) >> l;
    bytes += (size_t)side * side * (sizeof(float2) + sizeof(float));
    if (l + 1 < a.levels) {
      const int sc = min(a.m, a.tile + 2 * a.halo) >> (l + 1);
      bytes += (size_t)sc * sc * sizeof(float);
    }
    bytes = (bytes + 15) & ~(size_t)15;
  }
  return bytes;
}

constexpr size_t kPrepTileSmemMax = 96 * 1024;

// ---------------------------------------------------------------------------
// One scan position per CTA.
template <int M>
__host__ __device__ constexpr size_t level_floats2(int l) {
  return (size_t)(M >> l) * ((M >> l) + 1);
}

template <int M>
__host__ __device__ inline size_t step_smem_elems(int levels) {
  size_t n = level_floats2<M>(0);
  for (int l = 1; l < levels; ++l) n += 2 * level_floats2<M>(l);
  return n;
}

// The step of the allocation-free entry point: a.amp holds the caller's
// intensities d_k in natural order and the amplitude sqrt(max(d, 0)) is formed
// on the fly; ordered combine, no verify mode.
template <int M>
__global__ void __launch_bounds__(StepThreads<M>::value) k_step(const StepArgs a) {
  constexpr int NT = StepThreads<M>::value;
  constexpr int S = M + 1;
  constexpr int N1 = FftPlan<M>::N1, N2 = FftPlan<M>::N2;
  extern __shared__ float2 sm[];
  __shared__ double redd[NT / 32];
  __shared__ float redf[NT / 32];
  const int tid = threadIdx.x;
  const int kb = blockIdx.x;
  int k = a.order[kb];
  if (!EMG_INB(k, a.n_pos, kBcOrder)) k = 0;
  const bool slot_ok = EMG_INB(kb, a.b, kBcPatchWrite);
  const int o_r = a.pos[2 * k], o_c = a.pos[2 * k + 1];
  float2* buf = sm;

  // a1: z_k = P_k z, psi = Q z_k, mu_k = max |z_k|^2
  float mu_l = 0.f;
  for (int p = tid; p < M * M; p += NT) {
    const int r = p / M, c = p % M;
    const float2 zk = gather_obj(a.object, a.n_rows, a.n_cols, o_r + r, o_c + c);
    buf[r * S + c] = cmul(a.probe[p], zk);
    mu_l = fmaxf(mu_l, cabs2(zk));
  }
  const float mu = block_max<NT>(mu_l, redf);

  // a2: Psi = F psi (rows, then column pass A)
  fft2_fwd_until_col_b<M, NT>(buf, tid);

  // a2 (column pass B) + a3: Psi' = a_k Psi / |Psi| (scaled by 1/M^2) + a4 start
  const float* amp = a.amp + (size_t)k * M * M;
  const float inv_m2 = 1.f / (float)(M * M);
  float acc = 0.f;
  for (int s = tid; s < M * N2; s += NT) {
    const int k2 = s / M, c = s % M;
    float2 v[N1];
#pragma unroll
    for (int i = 0; i < N1; ++i) v[i] = buf[(i + N1 * k2) * S + c];
    Dft<N1, false>::run(v);
#pragma unroll
    for (int i = 0; i < N1; ++i) {
      const float am = sqrtf(fmaxf(amp[storage_to_freq<M>(i + N1 * k2) * M + storage_to_freq<M>(c)], 0.f));
      const float p2 = cabs2(v[i]);
      if (p2 > 0.f) {
        const float inv = rsqrtf(p2);
        const float dm = fmaf(p2, inv, -am);
        acc = fmaf(dm, dm, acc);
        v[i] = cscale(v[i], am * inv * inv_m2);
      } else {
        acc = fmaf(am, am, acc);
        v[i] = make_float2(am * inv_m2, 0.f);
      }
    }
    Dft<N1, true>::run(v);
#pragma unroll
    for (int i = 0; i < N1; ++i) buf[(i + N1 * k2) * S + c] = v[i];
  }
  __syncthreads();
  // a4: R = F^-1 Psi' (natural order)
  fft2_inv_after_col_b<M, NT>(buf, tid);
  const double phi = block_sum<NT>((double)acc, redd) * (0.5 / (double)(M * M));

  // a5: MAGPIE multigrid object step, patch-local (levels > 1)
  float2* Zl[kMaxLevels];
  float2* Rl[kMaxLevels];
  {
    size_t off = level_floats2<M>(0);
    for (int l = 1; l < a.levels; ++l) {
      Zl[l] = sm + off;
      off += level_floats2<M>(l);
      Rl[l] = sm + off;
      off += level_floats2<M>(l);
    }
  }
  if (a.levels > 1) {
    // restrict level 0 -> 1: z_1 = I_h^H (W_z z_k), R_1 = I_h^H (W_R R)
    {
      constexpr int mc = M / 2, sc = mc + 1;
      const float* Wz = a.lv.Wz[0];
      const float2* WR = a.lv.WR[0];
      for (int p = tid; p < mc * mc; p += NT) {
        const int i = p / mc, j = p % mc;
        float2 zs = czero(), rs = czero();
#pragma unroll
        for (int dy = 0; dy < 2; ++dy)
#pragma unroll
          for (int dx = 0; dx < 2; ++dx) {
            const int r = 2 * i + dy, c = 2 * j + dx;
            const float2 zk = gather_obj(a.object, a.n_rows, a.n_cols, o_r + r, o_c + c);
            zs = cadd(zs, cscale(zk, Wz[r * M + c]));
            rs = cadd(rs, cmul(WR[r * M + c], buf[r * S + c]));
          }
        Zl[1][i * sc + j] = cscale(zs, 0.25f);
        Rl[1][i * sc + j] = cscale(rs, 0.25f);
      }
    }
    __syncthreads();
    for (int l = 1; l + 1 < a.levels; ++l) {
      const int mf = M >> l, sf = mf + 1, mc = mf >> 1, sc = mc + 1;
      const float* Wz = a.lv.Wz[l];
      const float2* WR = a.lv.WR[l];
      for (int p = tid; p < mc * mc; p += NT) {
        const int i = p / mc, j = p % mc;
        float2 zs = czero(), rs = czero();
#pragma unroll
        for (int dy = 0; dy < 2; ++dy)
#pragma unroll
          for (int dx = 0; dx < 2; ++dx) {
            const int r = 2 * i + dy, c = 2 * j + dx;
            zs = cadd(zs, cscale(Zl[l][r * sf + c], Wz[r * mf + c]));
            rs = cadd(rs, cmul(WR[r * mf + c], Rl[l][r * sf + c]));
          }
        Zl[l + 1][i * sc + j] = cscale(zs, 0.25f);
        Rl[l + 1][i * sc + j] = cscale(rs, 0.25f);
      }
      __syncthreads();
    }
    // coarsest level: correction c = G (R - Q z), stored over z
    {
      const int l = a.levels - 1;
      const int ml = M >> l, sl = ml + 1;
      const float2* G = a.lv.G[l];
      const float2* Q = a.lv.Q[l];
      for (int p = tid; p < ml * ml; p += NT) {
        const int i = p / ml, j = p % ml;
        const float2 z = Zl[l][i * sl + j];
        Zl[l][i * sl + j] = cmul(G[p], csub(Rl[l][i * sl + j], cmul(Q[p], z)));
      }
      __syncthreads();
    }
    // back up: c_l = I_H^h c_{l+1} + G_l (R_l - Q_l (z_l + I_H^h c_{l+1}))
    for (int l = a.levels - 2; l >= 1; --l) {
      const int ml = M >> l, sl = ml + 1, mc = ml >> 1, sc = mc + 1;
      const float2* G = a.lv.G[l];
      const float2* Q = a.lv.Q[l];
      for (int p = tid; p < ml * ml; p += NT) {
        const int i = p / ml, j = p % ml;
        const float2 pro = prolong_at<float2>(Zl[l + 1], sc, mc, i, j, a.prolong);
        const float2 zp = cadd(Zl[l][i * sl + j], pro);
        Zl[l][i * sl + j] = cadd(pro, cmul(G[p], csub(Rl[l][i * sl + j], cmul(Q[p], zp))));
      }
      __syncthreads();
    }
  }

  // a5 (finest level) + a6 + a7: z+, Q+, geometric-mean joint step
  const float inv_mu = mu > 0.f ? 1.f / mu : 0.f;
  const float2* G0 = a.lv.G[0];
  float2* zt = a.zt + (size_t)kb * M * M;
  float2* qt = a.qt + (size_t)kb * M * M;
  for (int p = tid; p < M * M; p += NT) {
    const int r = p / M, c = p % M;
    const float2 zk = gather_obj(a.object, a.n_rows, a.n_cols, o_r + r, o_c + c);
    const float2 q = a.probe[p];
    const float2 R = buf[r * S + c];
    const float2 res = csub(R, cmul(q, zk));
    float2 zplus;
    if (a.levels == 1) {
      zplus = cadd(zk, cmul(G0[p], res));
    } else {
      constexpr int mc = M / 2, sc = mc + 1;
      const float2 pro = prolong_at<float2>(Zl[1], sc, mc, r, c, a.prolong);
      const float2 zp = cadd(zk, pro);
      zplus = cadd(zp, cmul(G0[p], csub(R, cmul(q, zp))));
    }
    const float2 qplus = cadd(q, cscale(cconjmul(zk, res), inv_mu));
    float2 zn, qn;
    if (a.joint) {
      zn = geometric_mean_aligned(zk, zplus);
      qn = geometric_mean_aligned(q, qplus);
    } else {
      zn = zplus;
      qn = qplus;
    }
    if (slot_ok) {
      zt[p] = zn;
      qt[p] = qn;
    }
  }
  if (tid == 0) {
    a.mu[kb] = mu;
    a.phi[kb] = phi;
  }
}

// ---------------------------------------------------------------------------
// One scan position per cluster of C CTAs (by default C = 1 for m <= 32, 2 for m = 64, 4 for
// m = 128, 8 for m = 256; also built: 2 for m <= 32, 4 for m = 64, 2 and 8 for m = 128).
//
// CTA `rank` owns patch rows [rank m/C, (rank+1) m/C) for the gather, the row
// FFT passes, the multigrid passes and the update, and storage columns
// [rank m/C, (rank+1) m/C) for the column FFT passes and the modulus
// replacement.  The two transposes between row and column slabs go through
// distributed shared memory; the multigrid up-pass reads the coarse rows
// adjacent to its slab from the neighbouring ranks (bilinear prolongation).
// The shared memory of a CTA is StepTile's.
namespace cg = cooperative_groups;

// Pixels per unrolled group in the update pass of the cluster step kernel.
#ifndef EMG_UPDATE_GROUP
#define EMG_UPDATE_GROUP 8
#endif

template <int M, int C>
struct CTile {
  static constexpr int H = M / C;              // rows of a row slab, columns of a column slab
  static constexpr int SR = M + 1;             // odd stride of a slab's lines: conflict-free
  static constexpr int N1 = FftPlan<M>::N1, N2 = FftPlan<M>::N2;
  static constexpr int NT = H * N1;            // one pass-A slot per thread
  static constexpr int PER = H * M / NT;       // slab pixels per thread
  static constexpr int SLOTS = H * N2 / NT;    // column pass-B slots per thread
  static_assert(H * M % NT == 0 && H * N2 % NT == 0 && NT <= 1024, "slab must split evenly");
  static_assert(H % N1 == 0, "the outputs of one pass-B slot go to one CTA");
};

// Shared memory of the step kernel.  A slab holds H lines of M elements (stride
// SR): my patch rows, or my storage columns, each line contiguous along the
// direction it is transformed in.
//
// ONE = false (m <= 128): a row slab, a column slab (later the multigrid
// buffers) and z_k on my rows.
// ONE = true (m = 256): one slab, overwritten in place by the transposes, and
// a second area that holds a_k on my storage columns during the transforms
// and the multigrid buffers after them; z_k is read again from L2 where the
// multigrid and the update need it.  199 KB per CTA with three slabs leave
// one CTA of 16 warps per SM and at most 15 clusters of 8 on the device (120
// SMs); 114 KB let two CTAs share an SM and hide each other's barriers.  An
// epoch of 4096 positions with minibatches of 256, when this was measured: 8.51
// -> 6.93 ms (with the transposes taken into the passes, which alone gave 0.428 ->
// 0.404 ms for 900 positions at m = 128 with minibatches of 64); 6.37 and 0.378 ms now.
template <int M, int C>
struct StepTile : CTile<M, C> {
  using B = CTile<M, C>;
  static constexpr int SIDE = M, CTAS = C;
  static constexpr bool ONE = M == 256;
  static constexpr int S = B::SR;
  // CTAs per SM the register budget leaves room for (as many as the shared memory does).  At m = 64
  // the cap pays where a minibatch fills the SMs several times over and costs where it does not (1444
  // positions, C = 2, three levels, us per epoch with it / without: minibatches of 1024 146 / 164, of 64
  // 343 / 332; two levels, of 256 182 / 187, of 64 with misfit 407 / 406).
  static constexpr int MIN_CTAS = ONE ? 2 : M == 128 ? C / 2 : M == 64 ? 3 * C / 2 : 1;
  static constexpr size_t slab = (size_t)B::H * S;
  // multigrid buffers of every level at which each CTA keeps a row
  static constexpr size_t mg_elems() {
    size_t n = 0;
    for (int w = M / 2; w >= C && w >= 2; w /= 2) n += (size_t)(2 * (w / C) + 2) * (w + 1);
    return n;
  }
  static constexpr size_t amp_elems = (size_t)B::H * M / 2;  // floats, counted in float2
  static constexpr size_t aux = mg_elems() > amp_elems ? mg_elems() : amp_elems;
  static constexpr size_t smem_elems = ONE ? slab + aux : 2 * slab + (size_t)B::H * M;
  static_assert(ONE || mg_elems() <= slab, "the multigrid buffers reuse the column slab");
};

// Forward and gradient kernels: whole launches of many positions, so the
// shared memory is one slab (transposed in place) and as many CTAs share an SM
// as 64 registers per thread allow.
// m = 128 fits one CTA of 1024 threads (no distributed shared memory): 900
// simulated positions 54 us against 64 with clusters of 2 and 62 with 4.  m = 256:
// clusters of 8 with two CTAs per SM 383 us for 1024 positions, of 4 with one 422.
template <int M> struct WaveCluster { static constexpr int value = M == 256 ? 8 : 1; };
template <int M, int C = WaveCluster<M>::value>
struct WaveTile : CTile<M, C> {
  using B = CTile<M, C>;
  static constexpr int SIDE = M, CTAS = C;
  static constexpr bool ONE = true;
  static constexpr int S = B::SR;
  static constexpr size_t slab = (size_t)B::H * S;
  static constexpr int MIN_CTAS = 1024 / B::NT;
  static_assert(B::H % B::N2 == 0, "the natural columns of one pass-B output index go to one CTA");
};

// Barrier of all CTAs of the cluster that also publishes shared-memory writes.
template <int C>
__device__ __forceinline__ void tile_sync(cg::cluster_group& cl) {
  if constexpr (C == 1)
    __syncthreads();
  else
    cl.sync();
}

// The same in two halves, so that register work between them hides the cluster
// barrier's latency (one CTA: the barrier is cheap and the wait does it all).
template <int C>
__device__ __forceinline__ void tile_arrive(cg::cluster_group& cl) {
  if constexpr (C > 1) cl.barrier_arrive();
}
template <int C>
__device__ __forceinline__ void tile_wait(cg::cluster_group& cl) {
  if constexpr (C == 1)
    __syncthreads();
  else
    cl.barrier_wait();
}

// `buf` of CTA d of the cluster.
template <int C, typename V>
__device__ __forceinline__ V* tile_rank(cg::cluster_group& cl, int rank, V* buf, int d) {
  if constexpr (C == 1)
    return buf;
  else
    return d == rank ? buf : cl.map_shared_rank(buf, d);
}

// Row pass B on my row slab, its outputs stored straight into the column slabs
// of all CTAs (the transpose costs no pass of its own).  Lanes take
// consecutive rows, which are consecutive elements of a column line, so each
// store of a warp is one contiguous run.  NAT = false: the slab of CTA d holds
// storage columns [d H, (d + 1) H); NAT = true: natural columns of that range.
// With one slab per CTA the outputs wait in registers until every CTA of the
// cluster has read its slab.  The caller's barrier makes the columns visible.
template <class T, bool NAT = false>
__device__ __forceinline__ void row_pass_b_to_cols(cg::cluster_group& cl, int rank, const float2* rowbuf,
                                                   float2* colbuf, int tid) {
  float2 v[T::SLOTS][T::N1];
  auto put = [&](int t) {
    const int s = tid + t * T::NT, k2 = s / T::H, at = rank * T::H + s % T::H;
    if constexpr (NAT) {
#pragma unroll
      for (int i = 0; i < T::N1; ++i) {
        const int d = T::N2 * i / T::H;  // k2 < N2 and N2 divides H
        tile_rank<T::CTAS>(cl, rank, colbuf, d)[(T::N2 * i % T::H + k2) * T::S + at] = v[t][i];
      }
    } else {
      const int e0 = T::N1 * k2;
      float2* dst = tile_rank<T::CTAS>(cl, rank, colbuf, e0 / T::H) + (e0 % T::H) * T::S + at;
#pragma unroll
      for (int i = 0; i < T::N1; ++i) dst[i * T::S] = v[t][i];
    }
  };
  auto get = [&](int t) {
    const int s = tid + t * T::NT;
    const float2* p = rowbuf + (s % T::H) * T::S + T::N1 * (s / T::H);
#pragma unroll
    for (int i = 0; i < T::N1; ++i) v[t][i] = p[i];
  };
  if constexpr (T::ONE) {
#pragma unroll
    for (int t = 0; t < T::SLOTS; ++t) get(t);
    tile_arrive<T::CTAS>(cl);  // I have read my slab
#pragma unroll
    for (int t = 0; t < T::SLOTS; ++t) Dft<T::N1, false>::run(v[t]);
    tile_wait<T::CTAS>(cl);
#pragma unroll
    for (int t = 0; t < T::SLOTS; ++t) put(t);
  } else {
#pragma unroll
    for (int t = 0; t < T::SLOTS; ++t) {
      get(t);
      Dft<T::N1, false>::run(v[t]);
      put(t);
    }
  }
}

// Inverse column pass A on my column slab, its outputs (natural rows) stored
// straight into the row slabs of all CTAs; lanes take consecutive columns,
// so each store of a warp is one contiguous run of a row.
template <class T>
__device__ __forceinline__ void col_pass_a_inv_to_rows(cg::cluster_group& cl, int rank, const float2* colbuf,
                                                       float2* rowbuf, int tid) {
  const int j = tid / T::H, line = tid % T::H;
  const float2* p = colbuf + line * T::S + j;
  float2 v[T::N2];
#pragma unroll
  for (int k2 = 0; k2 < T::N2; ++k2) v[k2] = p[T::N1 * k2];
  if constexpr (T::ONE) tile_arrive<T::CTAS>(cl);  // I have read my slab
#pragma unroll
  for (int k2 = 1; k2 < T::N2; ++k2) v[k2] = cmulc(v[k2], stage_twiddle<T::SIDE>(j, k2));
  Dft<T::N2, true>::run(v);
  if constexpr (T::ONE) tile_wait<T::CTAS>(cl);
#pragma unroll
  for (int n2 = 0; n2 < T::N2; ++n2) {
    const int d = T::N1 * n2 / T::H, lr = T::N1 * n2 % T::H + j;
    tile_rank<T::CTAS>(cl, rank, rowbuf, d)[lr * T::S + rank * T::H + line] = v[n2];
  }
}

// Writes v into slot [rank] of `arr` in every CTA of the cluster.
template <int C, typename V>
__device__ __forceinline__ void cluster_publish(cg::cluster_group& cl, int rank, V* arr, V v) {
#pragma unroll
  for (int d = 0; d < C; ++d) *tile_rank<C>(cl, rank, &arr[rank], d) = v;
}

// (I_H^h y)(lr, c) for a coarse row slab stored with one halo row above and
// below (y points at my first row, row stride sl); lr is the local fine row.
template <typename T>
__device__ __forceinline__ T prolong_halo(const T* y, int sl, int wc, int lr, int c, int kind) {
  const int i = lr >> 1, j = c >> 1;
  const T v = y[i * sl + j];
  if (kind == 0) return v;
  const int i2 = (lr & 1) ? i + 1 : i - 1;
  const int j2 = (c & 1) ? min(j + 1, wc - 1) : max(j - 1, 0);
  return lerp4<T>(v, y[i2 * sl + j], y[i * sl + j2], y[i2 * sl + j2]);
}

// Stores coarse value v of local row i, column j (a slab of hl rows, row stride
// sl, y at my first row) where the halo rows of the prolongation read it: my
// first row into the upper neighbour's bottom halo row (my own top halo row
// at the patch's top edge), my last row into the lower neighbour's top halo
// row (my own bottom halo row at the bottom edge).  A cluster barrier makes
// the rows visible before they are read.
template <int C, typename T>
__device__ __forceinline__ void push_halo(cg::cluster_group& cl, int rank, T* y, int sl, int hl, int i, int j, T v) {
  if constexpr (C == 1) {
    if (i == 0) y[j - sl] = v;
    if (i == hl - 1) y[hl * sl + j] = v;
  } else {
    if (i == 0) *(rank > 0 ? cl.map_shared_rank(y, rank - 1) + hl * sl + j : y - sl + j) = v;
    if (i == hl - 1) *(rank < C - 1 ? cl.map_shared_rank(y, rank + 1) - sl + j : y + hl * sl + j) = v;
  }
}

// One column of the object under a patch: pixel rows below (row0, col), 0 outside.
struct ObjectColumn {
  const float2* base;  // only dereferenced where the pixel exists
  int row0, n_rows, n_cols;
  bool col_ok;
  __device__ __forceinline__ ObjectColumn(const float2* object, int rows, int cols, int r, int c)
      : base(object + ((ptrdiff_t)r * cols + c)), row0(r), n_rows(rows), n_cols(cols),
        col_ok((unsigned)c < (unsigned)cols) {}
  __device__ __forceinline__ float2 at(int dr) const {
    if (col_ok && (unsigned)(row0 + dr) < (unsigned)n_rows) return base[(ptrdiff_t)dr * n_cols];
    return czero();
  }
};

// I_H^h at fine pixel (r, c) and at the pixels an even number of rows below it,
// from a coarse row slab with one halo row on each side (y: my first row).
struct CoarseCell {
  const float2* y;
  int dn, dj;  // offsets of the vertical and horizontal neighbours
  __device__ __forceinline__ CoarseCell(const float2* z, int stride, int width, int r, int c)
      : y(z + (r >> 1) * stride + (c >> 1)), dn((r & 1) ? stride : -stride),
        dj((c & 1) ? ((c >> 1) + 1 < width ? 1 : 0) : ((c >> 1) > 0 ? -1 : 0)) {}
  __device__ __forceinline__ float2 at(int off, bool bilinear) const {
    const float2* p = y + off;
    const float2 v = p[0];
    if (!bilinear) return v;
    return lerp4<float2>(v, p[dn], p[dj], p[dn + dj]);
  }
};

// The same at the pixel pair (r, c), (r, c + 1), c even: rows and centre column shared.
struct CoarsePair {
  const float2* y;
  int dn, jm, jp;
  __device__ __forceinline__ CoarsePair(const float2* z, int stride, int width, int r, int c)
      : y(z + (r >> 1) * stride + (c >> 1)), dn((r & 1) ? stride : -stride), jm((c >> 1) > 0 ? -1 : 0),
        jp((c >> 1) + 1 < width ? 1 : 0) {}
  __device__ __forceinline__ void at(int off, bool bilinear, float2 (&pro)[2]) const {
    const float2* p = y + off;
    const float2 v = p[0];
    if (!bilinear) {
      pro[0] = pro[1] = v;
      return;
    }
    const float2 w = p[dn];
    pro[0] = lerp4<float2>(v, w, p[jm], p[dn + jm]);
    pro[1] = lerp4<float2>(v, w, p[jp], p[dn + jp]);
  }
};

// RIN = true: the revised exit waves R_k and the misfit partials come from the
// tensor-core DFT pair (a2-a4 done elsewhere); the kernel gathers z_k and runs
// a5-a7 only.
template <int M, int C, bool RIN = false>
__global__ void __launch_bounds__(StepTile<M, C>::NT, StepTile<M, C>::MIN_CTAS) k_stepc(const StepArgs a) {
  using TL = StepTile<M, C>;
  constexpr bool ONE = TL::ONE;
  constexpr int NT = TL::NT, H = TL::H, SR = TL::S;
  constexpr int N1 = TL::N1, PER = TL::PER, SLOTS = TL::SLOTS;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = C == 1 ? 0 : (int)cl.block_rank();
  extern __shared__ __align__(16) float2 sm[];  // 16-byte aligned: the update pass reads pixel pairs
  float2* rowbuf = sm;                                        // my patch rows
  float2* colbuf = ONE ? sm : sm + TL::slab;                  // my storage columns (all rows)
  float2* mgbuf = ONE ? sm + TL::slab : colbuf;               // multigrid buffers, after the transforms
  float* ampbuf = reinterpret_cast<float*>(sm + TL::slab);    // ONE: a_k on my columns, [M][H], before them
  float2* zbuf = sm + 2 * TL::slab;                           // !ONE: H x M, z_k on my rows (gathered once)
  __shared__ float xf[C];
  __shared__ double xd[C], xd2[C];
  __shared__ double redd[2];
  __shared__ float redf[NT / 32];
  __shared__ int ticket_sh;
  // Phi_k of small probes: the threads' partials are added in FP64 (few warps, so the FP64
  // pipe's two results per clock and SM suffice); larger ones in FP32 warp trees.
  constexpr bool kSum64 = M <= 32;
  using Part = std::conditional_t<kSum64, double, float>;
  __shared__ double red64[kSum64 ? NT / 32 : 1];
  Part* sums;
  if constexpr (kSum64)
    sums = red64;
  else
    sums = redf;
  const int tid = threadIdx.x;
  int kb = blockIdx.x / C;
  if constexpr (!RIN) {
    if (a.prep_clusters > 0) {
      // role by ticket, taken before this launch lets the next one start: a
      // cluster only ever waits for clusters that started before it
      if (rank == 0 && tid == 0) ticket_sh = (int)(atomicAdd(a.sync, 1u) - a.ticket_base);
      tile_sync<C>(cl);  // every CTA of the cluster is running; rank 0's ticket is visible
      const int t = *tile_rank<C>(cl, rank, &ticket_sh, 0);
      if (t < a.prep_clusters) {
        pdl_trigger();
        pdl_wait();  // the probe and max|Q|^2 come from the previous combine
        const int tile = t * C + rank;
        if (tile < a.prep_tiles) {
          prep_tile_body(a.prep, tile, tid, NT, sm);
          __syncthreads();
          if (tid == 0) {
            __threadfence();
            atomicAdd(a.sync + 1, 1u);
          }
        }
        if constexpr (C > 1) cl.sync();  // no CTA leaves while a peer may still read rank 0's ticket
        return;
      }
      kb = t - a.prep_clusters;
    }
  }
  int k = a.order[kb];
  if (!EMG_INB(k, a.n_pos, kBcOrder)) k = 0;
  const bool slot_ok = EMG_INB(kb, a.b, kBcPatchWrite);
  const int o_r = a.pos[2 * k], o_c = a.pos[2 * k + 1];
  const int row0 = rank * H;

  // amplitudes of my spectral slots: issued now, consumed after the row passes
  float am_reg[ONE ? 1 : SLOTS][ONE ? 1 : N1];
  if constexpr (!RIN) {
    const float* amp = a.amp + (size_t)k * M * M + rank * H;
    if constexpr (ONE) {
#pragma unroll
      for (int q = tid; q < M * H / 4; q += NT)
        cp_async16(ampbuf + 4 * q, amp + (q / (H / 4)) * M + 4 * (q % (H / 4)));
      cp_async_commit();
    } else {
#pragma unroll
      for (int t = 0; t < SLOTS; ++t) {
        const int s = tid + t * NT, k2 = s / H, lc = s % H;
#pragma unroll
        for (int i = 0; i < N1; ++i) am_reg[t][i] = __ldg(amp + (i + N1 * k2) * M + lc);
      }
    }
  }
  pdl_trigger();
  pdl_wait();  // object, probe, max|Q|^2 and level arrays come from earlier kernels
  const float MQ = __uint_as_float(*a.mq);
  if constexpr (C > 1) cluster_arrive_relaxed();  // completed (wait) before the first distributed shared memory access

  // a1: gather my rows, psi = Q z_k, partial mu_k
  float mu_l = 0.f;
  // pixels of a thread whose gather loads are in flight together (more costs
  // registers that the small tiles need for their occupancy; m = 256: all 16, 6.37 ms per
  // epoch of 4096 positions against 6.51 with 8 and 6.53 with 4)
#ifdef EMG_GATHER_UNROLL
  constexpr int kGatherUnroll = EMG_GATHER_UNROLL;
#else
  constexpr int kGatherUnroll = ONE ? 16 : M >= 128 ? 8 : 4;
#endif
  // A thread's pixels lie in one column, RPT rows apart (NT is a multiple of M),
  // so every address is a base of the thread plus a constant per pixel.
  constexpr int RPT = NT / M;
  static_assert(NT % M == 0, "a thread's pixels share one column");
  {
    const int l0 = tid / M, c0 = tid % M;
    const ObjectColumn zc(a.object, a.n_rows, a.n_cols, o_r + row0 + l0, o_c + c0);
    float2* rb = rowbuf + l0 * SR + c0;
    const float2* src = RIN ? a.r_in + (size_t)kb * M * M : a.probe;
    src += row0 * M + tid;
#pragma unroll (kGatherUnroll)
    for (int t = 0; t < PER; ++t) {
      const float2 zk = zc.at(t * RPT);
      if constexpr (!ONE) zbuf[tid + t * NT] = zk;
      const float2 x = src[t * NT];
      rb[t * RPT * SR] = RIN ? x : cmul(x, zk);
      mu_l = fmaxf(mu_l, cabs2(zk));
    }
  }
  // per-warp maxima of |z_k|^2; the barrier also orders the gather before the row passes
  warp_partial_max(mu_l, redf);
  __syncthreads();
  if constexpr (!RIN) {
    // a2: row pass A on my rows
    gpass_a_fwd<M, H, SR, 1, NT>(rowbuf, tid);
    if constexpr (ONE) cp_async_wait_all();  // a_k; the barriers below show it to the whole CTA
    __syncthreads();
  }
  if constexpr (C > 1) cl.barrier_wait();  // all CTAs of the cluster resident
  // row pass B, outputs to the column slabs
  if constexpr (!RIN) row_pass_b_to_cols<TL>(cl, rank, rowbuf, colbuf, tid);
  if (tid == 0) cluster_publish<C>(cl, rank, xf, partials_max<NT>(redf));
  tile_sync<C>(cl);
  float mu = xf[0];
#pragma unroll
  for (int d = 1; d < C; ++d) mu = fmaxf(mu, xf[d]);

  if constexpr (!RIN) {
  // a2 (columns) + a3 + a4 (columns) on my storage columns
  gpass_a_fwd<M, H, SR, 1, NT>(colbuf, tid);
  __syncthreads();
  const float inv_m2 = 1.f / (float)(M * M);
  float acc = 0.f;
#pragma unroll
  for (int t = 0; t < SLOTS; ++t) {
    const int s = tid + t * NT, k2 = s / H, lc = s % H;
    float2* p = colbuf + lc * SR + N1 * k2;
    float2 v[N1];
#pragma unroll
    for (int i = 0; i < N1; ++i) v[i] = p[i];
    Dft<N1, false>::run(v);
#pragma unroll
    for (int i = 0; i < N1; ++i) {
      float am;
      if constexpr (ONE)
        am = ampbuf[(i + N1 * k2) * H + lc];
      else
        am = am_reg[t][i];
      const float p2 = cabs2(v[i]);
      if (p2 > 0.f) {
        const float inv = rsqrtf(p2);
        const float dm = fmaf(p2, inv, -am);
        acc = fmaf(dm, dm, acc);
        v[i] = cscale(v[i], am * inv * inv_m2);
      } else {
        acc = fmaf(am, am, acc);
        v[i] = make_float2(am * inv_m2, 0.f);
      }
    }
    Dft<N1, true>::run(v);
#pragma unroll
    for (int i = 0; i < N1; ++i) p[i] = v[i];
  }
  // per-warp misfit partials; the barrier also orders the pass before the next one
  warp_partial_sum<Part>(acc, sums);
  __syncthreads();
  // inverse column pass A, outputs to the row slabs
  col_pass_a_inv_to_rows<TL>(cl, rank, colbuf, rowbuf, tid);
  if (tid == 0) cluster_publish<C>(cl, rank, xd, partials_sum<NT>(sums));
  tile_sync<C>(cl);
  // a4: inverse row passes -> R (natural order) on my rows
  gpass_b<M, H, SR, 1, NT, true>(rowbuf, tid);
  __syncthreads();
  gpass_a_inv<M, H, SR, 1, NT>(rowbuf, tid);
  __syncthreads();
  }  // !RIN

  if constexpr (!RIN) {
    if (a.prep_clusters > 0) {
      // the level arrays of this minibatch (with one level the gain G_0 alone) come
      // from the prep clusters of this launch
      if (tid == 0) {
        const unsigned long long t0 = globaltimer_ns();
        while (ld_acquire_u32(a.sync + 1) < a.prep_target) {
          if (globaltimer_ns() - t0 > kFusedPrepWaitNs) {
            atomicExch(a.sync + 2, 1u);
            break;
          }
        }
      }
      __syncthreads();
    }
  }
  // a5: MAGPIE multigrid on row slabs; level-l buffers (l >= 1) in mgbuf.
  // Z_l keeps one halo row above and below my rows for the prolongation.
  const bool halo = a.prolong != 0;
  constexpr int W1 = M / 2, H1 = W1 / C, S1 = W1 + 1;  // level 1: width, my rows, row stride
  constexpr int W2 = M / 4, H2 = W2 / C, S2 = W2 + 1;  // level 2
  float2* const Z1 = mgbuf + S1;
  float2* const R1 = mgbuf + (H1 + 2) * S1;
  float2* const Z2 = R1 + H1 * S1 + S2;
  // Level-1 pixels of a thread: one column, RP1 rows apart (even, so the
  // prolongation's neighbours lie on the same side for all of them).
  constexpr int P1 = H1 * W1 / NT, RP1 = NT / W1;
  static_assert(H1 * W1 % NT == 0 && NT % W1 == 0 && RP1 % 2 == 0, "level 1 splits evenly over the threads");
  const int i1 = tid / W1, j1 = tid % W1;
  // Level-2 pixels; where a slab has fewer than NT of them the other threads have none.
  constexpr bool kHas2 = H2 >= 1 && (H2 * W2 % NT == 0 || H2 * W2 < NT);
  constexpr int P2 = kHas2 && H2 * W2 >= NT ? H2 * W2 / NT : 1, RP2 = NT / W2;
  const int i2 = tid / W2, j2 = tid % W2;
  const bool on2 = H2 * W2 >= NT || tid < H2 * W2;
  // With two levels the coarse step follows the restriction at the same pixel
  // at once (it needs nothing from other threads).  With three levels every
  // level array the coarse levels need is loaded into registers beside the
  // loads of the first restriction, so the coarse phases wait on no load
  // (ONE: where they are used; the other CTA of the SM covers the wait and the
  // registers are not there to hold them).  More levels take the general loops.
  const bool l3 = kHas2 && a.levels == 3;
  // Copies the rows of the coarse correction at level l (Z: my first row) adjacent
  // to my slab (from the neighbouring ranks, or my own edge row where the patch ends).
  auto fill_halo = [&](float2* Z, int l) {
    const int wl = M >> l, hl = wl / C, sl = wl + 1;
    const float2* Zup = Z;
    const float2* Zdn = Z;
    if constexpr (C > 1) {
      if (rank > 0) Zup = cl.map_shared_rank(Z, rank - 1);
      if (rank < C - 1) Zdn = cl.map_shared_rank(Z, rank + 1);
    }
    for (int j = tid; j < wl; j += NT) {
      Z[-sl + j] = rank > 0 ? Zup[(hl - 1) * sl + j] : Z[j];
      Z[hl * sl + j] = rank < C - 1 ? Zdn[j] : Z[(hl - 1) * sl + j];
    }
  };
  // Levels 1 .. L - 1 for any L, from Z_1 and R_1 to the correction at level 1.
  auto general_levels = [&]() {
    float2* Zl[kMaxLevels];
    float2* Rl[kMaxLevels];
    size_t off = 0;
    for (int l = 1; l < a.levels; ++l) {
      const int wl = M >> l, hl = wl / C, sl = wl + 1;
      Zl[l] = mgbuf + off + sl;
      off += (size_t)(hl + 2) * sl;
      Rl[l] = mgbuf + off;
      off += (size_t)hl * sl;
    }
    for (int l = 1; l + 1 < a.levels; ++l) {
      const int wf = M >> l, sf = wf + 1, hf = wf / C, wc = wf >> 1, hc = wc / C, sc = wc + 1;
      const float* Wz = a.lv.Wz[l];
      const float2* WR = a.lv.WR[l];
      const float2* __restrict__ const Zf = Zl[l];
      const float2* __restrict__ const Rf = Rl[l];
      float2* __restrict__ const Zc = Zl[l + 1];
      float2* __restrict__ const Rc = Rl[l + 1];
      for (int p = tid; p < hc * wc; p += NT) {
        const int i = p / wc, j = p % wc;
        float2 zs = czero(), rs = czero();
#pragma unroll
        for (int dy = 0; dy < 2; ++dy)
#pragma unroll
          for (int dx = 0; dx < 2; ++dx) {
            const int lr = 2 * i + dy, r = rank * hf + lr, c = 2 * j + dx;
            const int wi = EMG_INB(r * wf + c, wf * wf, kBcLevel) ? r * wf + c : 0;
            zs = cadd(zs, cscale(Zf[lr * sf + c], __ldcg(Wz + wi)));
            rs = cadd(rs, cmul(__ldcg(WR + wi), Rf[lr * sf + c]));
          }
        Zc[i * sc + j] = cscale(zs, 0.25f);
        Rc[i * sc + j] = cscale(rs, 0.25f);
      }
      __syncthreads();
    }
    {  // coarsest level: correction c = G (R - Q z), stored over z
      const int l = a.levels - 1;
      const int wl = M >> l, hl = wl / C, sl = wl + 1;
      const float2* G = a.lv.G[l];
      const float2* Q = a.lv.Q[l];
      float2* __restrict__ const Zw = Zl[l];
      const float2* __restrict__ const Rw = Rl[l];
      for (int p = tid; p < hl * wl; p += NT) {
        const int i = p / wl, j = p % wl, gi = rank * hl + i;
        const int li = EMG_INB(gi * wl + j, wl * wl, kBcLevel) ? gi * wl + j : 0;
        const float2 z = Zw[i * sl + j];
        Zw[i * sl + j] = cmul(__ldcg(G + li), csub(Rw[i * sl + j], cmul(__ldcg(Q + li), z)));
      }
    }
    // back up: c_l = I_H^h c_{l+1} + G_l (R_l - Q_l (z_l + I_H^h c_{l+1}))
    for (int l = a.levels - 2; l >= 1; --l) {
      if (halo) {
        tile_sync<C>(cl);
        fill_halo(Zl[l + 1], l + 1);
      }
      __syncthreads();
      const int wl = M >> l, hl = wl / C, sl = wl + 1, wc = wl >> 1, sc = wc + 1;
      const float2* G = a.lv.G[l];
      const float2* Q = a.lv.Q[l];
      float2* __restrict__ const Zw = Zl[l];
      const float2* __restrict__ const Rw = Rl[l];
      const float2* __restrict__ const Zc = Zl[l + 1];
#pragma unroll 4
      for (int p = tid; p < hl * wl; p += NT) {
        const int i = p / wl, j = p % wl, gi = rank * hl + i;
        const int li = EMG_INB(gi * wl + j, wl * wl, kBcLevel) ? gi * wl + j : 0;
        const float2 pro = prolong_halo<float2>(Zc, sc, wc, i, j, a.prolong);
        const float2 zp = cadd(Zw[i * sl + j], pro);
        Zw[i * sl + j] = cadd(pro, cmul(__ldcg(G + li), csub(Rw[i * sl + j], cmul(__ldcg(Q + li), zp))));
      }
    }
  };
  if (a.levels > 1) {
    float2 pf_wz1[P2][2];     // W_z,1 at (2i + dy, 2j .. 2j + 1): (dx 0, dx 1) per dy
    float4 pf_wr1[P2][2];     // W_R,1 at the same pixels
    float2 pf_g2[P2], pf_q2[P2], pf_g1[P1], pf_q1[P1];
    auto load_down = [&]() {
#pragma unroll
      for (int t = 0; t < P2; ++t) {
        if (!on2) break;
        const int i = i2 + t * RP2, wb = (rank * H1 + 2 * i) * W1 + 2 * j2, lb = (rank * H2 + i) * W2 + j2;
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
          const int wi = EMG_INB(wb + dy * W1 + 1, W1 * W1, kBcLevel) ? wb + dy * W1 : 0;
          pf_wz1[t][dy] = __ldcg(reinterpret_cast<const float2*>(a.lv.Wz[1] + wi));
          pf_wr1[t][dy] = __ldcg(reinterpret_cast<const float4*>(a.lv.WR[1] + wi));
        }
        const int li = EMG_INB(lb, W2 * W2, kBcLevel) ? lb : 0;
        pf_g2[t] = __ldcg(a.lv.G[2] + li);
        pf_q2[t] = __ldcg(a.lv.Q[2] + li);
      }
    };
    auto load_up = [&]() {
#pragma unroll
      for (int t = 0; t < P1; ++t) {
        const int lb = rank * H1 * W1 + tid + t * NT;
        const int li = EMG_INB(lb, W1 * W1, kBcLevel) ? lb : 0;
        pf_g1[t] = __ldcg(a.lv.G[1] + li);
        pf_q1[t] = __ldcg(a.lv.Q[1] + li);
      }
    };
    // restrict level 0 -> 1: z_1 = I_h^H (W_z z_k), R_1 = I_h^H (W_R R); with
    // two levels at once the coarsest step c = G (R - Q z)
    auto restrict_top = [&](auto two_levels) {
      constexpr bool kTwo = decltype(two_levels)::value;
      const int f0 = 2 * i1, c0 = 2 * j1;  // fine pixel of the first coarse one, 2 RP1 rows apart
      const float* Wz = a.lv.Wz[0] + (row0 + f0) * M + c0;
      const float2* WR = a.lv.WR[0] + (row0 + f0) * M + c0;
      const float2* rb = rowbuf + f0 * SR + c0;
      const ObjectColumn za(a.object, a.n_rows, a.n_cols, o_r + row0 + f0, o_c + c0);
      const ObjectColumn zb(a.object, a.n_rows, a.n_cols, o_r + row0 + f0, o_c + c0 + 1);
      float2* zw = Z1 + i1 * S1 + j1;
      float2* rw = R1 + i1 * S1 + j1;
#pragma unroll
      for (int t = 0; t < P1; ++t) {
        float2 zs = czero(), rs = czero();
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
          const int fr = 2 * RP1 * t + dy;
          // the weights of the pixel pair (c, c + 1) in one load each (c is even)
          const float2 wz = __ldcg(reinterpret_cast<const float2*>(Wz + fr * M));
          const float4 wr = __ldcg(reinterpret_cast<const float4*>(WR + fr * M));
          float2 z0, z1;
          if constexpr (ONE) {
            z0 = za.at(fr);
            z1 = zb.at(fr);
          } else {
            z0 = zbuf[(f0 + fr) * M + c0];
            z1 = zbuf[(f0 + fr) * M + c0 + 1];
          }
          zs = cadd(zs, cscale(z0, wz.x));
          rs = cfma(make_float2(wr.x, wr.y), rb[fr * SR], rs);
          zs = cadd(zs, cscale(z1, wz.y));
          rs = cfma(make_float2(wr.z, wr.w), rb[fr * SR + 1], rs);
        }
        const float2 z1 = cscale(zs, 0.25f), r1 = cscale(rs, 0.25f);
        if constexpr (kTwo) {
          const float2 cc = cmul(pf_g1[t], cfnma(pf_q1[t], z1, r1));
          zw[t * RP1 * S1] = cc;
          if (halo) push_halo<C>(cl, rank, Z1, S1, H1, i1 + t * RP1, j1, cc);
        } else {
          zw[t * RP1 * S1] = z1;
          rw[t * RP1 * S1] = r1;
        }
      }
    };
    if (a.levels == 2) {
      load_up();
      restrict_top(std::true_type{});
    } else {
      if (!ONE && l3) {
        load_down();
        load_up();
      }
      restrict_top(std::false_type{});
      __syncthreads();
      if (l3) {
        if (ONE) load_down();
        // restrict 1 -> 2 and at once the coarsest step on the same level-2 pixel
        if (on2) {
          const float2* zf = Z1 + 2 * i2 * S1 + 2 * j2;
          const float2* rf = R1 + 2 * i2 * S1 + 2 * j2;
          float2* zw = Z2 + i2 * S2 + j2;
#pragma unroll
          for (int t = 0; t < P2; ++t) {
            float2 zs = czero(), rs = czero();
#pragma unroll
            for (int dy = 0; dy < 2; ++dy) {
              const int at = (2 * RP2 * t + dy) * S1;
              zs = cadd(zs, cscale(zf[at], pf_wz1[t][dy].x));
              rs = cfma(make_float2(pf_wr1[t][dy].x, pf_wr1[t][dy].y), rf[at], rs);
              zs = cadd(zs, cscale(zf[at + 1], pf_wz1[t][dy].y));
              rs = cfma(make_float2(pf_wr1[t][dy].z, pf_wr1[t][dy].w), rf[at + 1], rs);
            }
            const float2 z2 = cscale(zs, 0.25f), r2 = cscale(rs, 0.25f);
            // coarsest level 2: correction c = G (R - Q z), stored over z
            const float2 cc = cmul(pf_g2[t], cfnma(pf_q2[t], z2, r2));
            zw[t * RP2 * S2] = cc;
            if (halo) push_halo<C>(cl, rank, Z2, S2, H2, i2 + t * RP2, j2, cc);
          }
        }
        if (ONE) load_up();
        if (halo)
          tile_sync<C>(cl);  // the pushed halo rows of level 2 are in place
        else
          __syncthreads();
        {  // back up to level 1
          const CoarseCell cell(Z2, S2, W2, i1, j1);
          float2* zw = Z1 + i1 * S1 + j1;
          const float2* rw = R1 + i1 * S1 + j1;
#pragma unroll
          for (int t = 0; t < P1; ++t) {
            const float2 pro = cell.at(t * (RP1 / 2) * S2, halo);
            const float2 zp = cadd(zw[t * RP1 * S1], pro);
            const float2 cc = cfma(pf_g1[t], cfnma(pf_q1[t], zp, rw[t * RP1 * S1]), pro);
            zw[t * RP1 * S1] = cc;
            if (halo) push_halo<C>(cl, rank, Z1, S1, H1, i1 + t * RP1, j1, cc);
          }
        }
      } else {
        general_levels();
      }
    }
    if (halo) tile_sync<C>(cl);
    const bool pushed = a.levels == 2 || l3;  // the halo rows of level 1 are in place
    if (halo && !pushed) fill_halo(Z1, 1);
    if (!halo || !pushed) __syncthreads();
  }

  // a5 (finest level) + a6 + a7; the level-0 gain G_0 = conj(Q)/(u_0 + |Q|^2)
  // comes from the probe prep of this minibatch
  const float inv_mu = mu > 0.f ? 1.f / mu : 0.f;
  float2* zt = a.zt + (size_t)kb * M * M;
  float2* qt = a.qt + (size_t)kb * M * M;
  const float2* G0 = a.lv.G[0];
  float acc_after = 0.f;
  // Groups of UG pixels: the probe and gain loads of a group are issued
  // together, and the loop body stays small enough for the instruction cache.
  // (two CTAs per SM at m = 256 hide the load latency and leave 64 registers: one pair at a
  // time, 6.51 ms per epoch of 4096 positions against 6.68 with groups of 4 and 7.14 with 8)
  constexpr int UGM = ONE ? 2 : EMG_UPDATE_GROUP;
  constexpr int UG0 = UGM < PER ? UGM : PER;
  constexpr int UG = PER % UG0 == 0 ? UG0 : 1;
  // The common case (ordered combine, no verify) runs a loop without the mode
  // branches over pairs of adjacent pixels, with 16-byte probe and gain loads
  // and patch stores, and the prolongation's loads shared by the pair; the
  // arithmetic per pixel is the same as in the general loop.  A thread's pairs
  // lie in one column pair, RP rows apart (even).
  constexpr int UGP = UG >= 2 && PER % 2 == 0 ? UG / 2 : 0;
  const bool pairs = UGP > 0 && !a.s_num && !a.verify && slot_ok &&
                     ((reinterpret_cast<uintptr_t>(a.probe) | reinterpret_cast<uintptr_t>(G0) |
                       reinterpret_cast<uintptr_t>(zt) | reinterpret_cast<uintptr_t>(qt)) & 15) == 0;
  // Small probes take the accuracy of correctly rounded roots, as the allocation-free step does: no
  // floor under the squares (an object in units of 1e-9 has |z z+|^2 of 1e-36), and at an exact tie the
  // principal root.  (An epoch of 100 positions at m = 32, minibatches of 10: 84 us, with IEEE roots and
  // division 107.)
  constexpr bool kRounded = M <= 32;
  auto update_pairs = [&](auto multigrid, auto joint) {
    constexpr bool kMg = decltype(multigrid)::value, kJoint = decltype(joint)::value;
    constexpr int PP = PER / 2, RP = 2 * RPT;
    const int l0 = 2 * tid / M, c0 = 2 * tid % M;
    const float2* rb = rowbuf + l0 * SR + c0;
    const ObjectColumn za(a.object, a.n_rows, a.n_cols, o_r + row0 + l0, o_c + c0);
    const ObjectColumn zb(a.object, a.n_rows, a.n_cols, o_r + row0 + l0, o_c + c0 + 1);
    const CoarsePair cell(Z1, S1, W1, l0, c0);
    const int off0 = row0 * M + 2 * tid;
#pragma unroll 1
    for (int t0 = 0; t0 < PP; t0 += UGP) {
      float4 qv[UGP], gv[UGP];
#pragma unroll
      for (int u = 0; u < UGP; ++u) {
        const int off = off0 + 2 * (t0 + u) * NT;
        qv[u] = __ldg(reinterpret_cast<const float4*>(a.probe + off));
        gv[u] = __ldcg(reinterpret_cast<const float4*>(G0 + off));
      }
      [[maybe_unused]] float4 zv[ONE ? UGP : 1];
      if constexpr (ONE) {
#pragma unroll
        for (int u = 0; u < UGP; ++u) {
          const float2 z0 = za.at((t0 + u) * RP), z1 = zb.at((t0 + u) * RP);
          zv[u] = make_float4(z0.x, z0.y, z1.x, z1.y);
        }
      }
#pragma unroll
      for (int u = 0; u < UGP; ++u) {
        const int t = t0 + u;
        float4 zk2;
        if constexpr (ONE)
          zk2 = zv[u];
        else
          zk2 = *reinterpret_cast<const float4*>(zbuf + 2 * tid + 2 * t * NT);
        // coarse-level correction at both pixels
        float2 pro[2] = {czero(), czero()};
        if constexpr (kMg) cell.at(t * (RP / 2) * S1, halo, pro);
        float2 zo[2], qo[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float2 zk = h ? make_float2(zk2.z, zk2.w) : make_float2(zk2.x, zk2.y);
          const float2 q = h ? make_float2(qv[u].z, qv[u].w) : make_float2(qv[u].x, qv[u].y);
          const float2 g0 = h ? make_float2(gv[u].z, gv[u].w) : make_float2(gv[u].x, gv[u].y);
          update_pixel<kMg, kJoint, kRounded>(zk, q, g0, rb[t * RP * SR + h], pro[h], inv_mu, zo[h], qo[h]);
        }
        const int off = off0 + 2 * t * NT;
        *reinterpret_cast<float4*>(zt + off) = make_float4(zo[0].x, zo[0].y, zo[1].x, zo[1].y);
        *reinterpret_cast<float4*>(qt + off) = make_float4(qo[0].x, qo[0].y, qo[1].x, qo[1].y);
      }
    }
  };
  if constexpr (UGP > 0) {
    if (pairs) {
      if (a.levels > 1) {
        if (a.joint)
          update_pairs(std::true_type{}, std::true_type{});
        else
          update_pairs(std::true_type{}, std::false_type{});
      } else {
        if (a.joint)
          update_pairs(std::false_type{}, std::true_type{});
        else
          update_pairs(std::false_type{}, std::false_type{});
      }
    }
  }
#pragma unroll 1
  for (int t0 = 0; t0 < (pairs ? 0 : PER); t0 += UG) {
  float2 qv[UG], gv[UG];
#pragma unroll
  for (int u = 0; u < UG; ++u) {
    qv[u] = __ldg(a.probe + row0 * M + tid + (t0 + u) * NT);
    gv[u] = __ldcg(G0 + row0 * M + tid + (t0 + u) * NT);
  }
#pragma unroll
  for (int u = 0; u < UG; ++u) {
    const int t = t0 + u;
    const int p = tid + t * NT;
    const int lr = p / M, c = p % M, r = row0 + lr;
    float2 zk;
    if constexpr (ONE)
      zk = gather_obj(a.object, a.n_rows, a.n_cols, o_r + r, o_c + c);
    else
      zk = zbuf[p];
    const float2 q = qv[u];
    const float2 R = rowbuf[lr * SR + c];
    const float2 pro = a.levels == 1 ? czero() : prolong_halo<float2>(Z1, S1, W1, lr, c, a.prolong);
    float2 zn, qn;
    if (a.levels == 1) {
      if (a.joint)
        update_pixel<false, true, kRounded>(zk, q, gv[u], R, pro, inv_mu, zn, qn);
      else
        update_pixel<false, false, kRounded>(zk, q, gv[u], R, pro, inv_mu, zn, qn);
    } else {
      if (a.joint)
        update_pixel<true, true, kRounded>(zk, q, gv[u], R, pro, inv_mu, zn, qn);
      else
        update_pixel<true, false, kRounded>(zk, q, gv[u], R, pro, inv_mu, zn, qn);
    }
    if (a.s_num)
      scatter_atomic(a.s_num, a.s_den, a.combine, a.n_rows, a.n_cols, o_r + r, o_c + c, zn, zk, fmaf(a.w_eps, MQ, cabs2(q)));
    else if (slot_ok)
      zt[r * M + c] = zn;
    if (slot_ok) qt[r * M + c] = qn;
    if (a.verify) acc_after += cabs2(csub(cmul(qn, zn), R));
  }
  }
  if (a.verify) {
    double part = 0.0;
    if constexpr (kSum64) {
      warp_partial_sum<Part>(acc_after, sums);
      __syncthreads();
      if (tid == 0) part = 0.5 * partials_sum<NT>(sums);
    } else {
      part = 0.5 * block_sum_f<NT>(acc_after, redf, redd);
    }
    if (tid == 0) cluster_publish<C>(cl, rank, xd2, part);
  }
  // With halo rows read from the neighbours (bilinear prolongation, other
  // than two or three levels) a neighbour may still read my coarse rows: no CTA leaves
  // before all arrive.  The verify mode also publishes xd2, which needs the
  // release / acquire pair.  Otherwise no CTA touches another's shared memory
  // after the last cluster barrier, and each may leave when done.
  if (a.verify) {
    tile_sync<C>(cl);
  } else if (C > 1 && halo && !l3 && a.levels > 2) {
    cluster_arrive_relaxed();
    cluster_wait();
  }
  if (rank == 0 && tid == 0) {
    double phi = 0.0, after = 0.0;
#pragma unroll
    for (int d = 0; d < C; ++d) {
      if constexpr (!RIN) phi += xd[d];
      after += xd2[d];
    }
    if constexpr (RIN)
      for (int t = 0; t < a.r_tiles; ++t) phi += a.r_partial[(size_t)kb * a.r_tiles + t];
    a.mu[kb] = mu;
    a.phi[kb] = phi * (0.5 / (double)(M * M));
    if (a.verify) a.phi_after[kb] = after;
  }
}

// ---------------------------------------------------------------------------
// Forward transform of one tile per cluster: modes
//   0 misfit partial (1/2 m^2) sum (|F psi| - a_k)^2 per position (Parseval
//     form of Eq. exit_misfit),
//   1 intensity |F psi|^2 in natural order (data model of Sec. 2.1),
//   2 F x of a natural-order tile, 3 F^-1 x = conj(F conj(x / m^2)).
// Bound by instruction issue and shared-memory latency, so the tile takes the
// smallest cluster whose slab leaves 32 warps per SM.  The outputs of modes
// 1-3 leave column pass B from registers: the slabs hold natural columns, so a
// warp writes whole 128-byte runs of a natural row.
template <int M, int MODE>
__global__ void __launch_bounds__(WaveTile<M>::NT, WaveTile<M>::MIN_CTAS) k_forward(const FwdArgs a) {
  using TL = WaveTile<M>;
  constexpr int NT = TL::NT, H = TL::H, S = TL::S, N1 = TL::N1, N2 = TL::N2, C = TL::CTAS, PER = TL::PER;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = C == 1 ? 0 : (int)cl.block_rank();
  extern __shared__ float2 sm[];
  __shared__ double xd[C];
  __shared__ double redd[(NT + 31) / 32];
  const int tid = threadIdx.x;
  const int t = blockIdx.x / C;
  const int row0 = rank * H;
  const float inv_m2 = 1.f / (float)(M * M);
  // a thread's pixels: one column, RPT rows apart
  constexpr int RPT = NT / M;
  static_assert(NT % M == 0, "a thread's pixels share one column");
  float2* mine = sm + (tid / M) * S + tid % M;
  if constexpr (MODE >= 2) {
    const float2* x = a.in + (size_t)t * M * M + row0 * M + tid;
#pragma unroll (PER < 8 ? PER : 8)
    for (int u = 0; u < PER; ++u) {
      const float2 v = x[u * NT];
      mine[u * RPT * S] = MODE == 3 ? make_float2(v.x * inv_m2, -v.y * inv_m2) : v;
    }
  } else {
    const int o_r = a.pos[2 * t], o_c = a.pos[2 * t + 1];
    const ObjectColumn zc(a.object, a.n_rows, a.n_cols, o_r + row0 + tid / M, o_c + tid % M);
    const float2* q = a.probe + row0 * M + tid;
#pragma unroll (PER < 8 ? PER : 8)
    for (int u = 0; u < PER; ++u) mine[u * RPT * S] = cmul(q[u * NT], zc.at(u * RPT));
  }
  __syncthreads();
  gpass_a_fwd<M, H, S, 1, NT>(sm, tid);
  __syncthreads();
  row_pass_b_to_cols<TL, MODE != 0>(cl, rank, sm, sm, tid);
  tile_sync<C>(cl);
  gpass_a_fwd<M, H, S, 1, NT>(sm, tid);
  __syncthreads();
  float acc = 0.f;
#pragma unroll
  for (int q = 0; q < TL::SLOTS; ++q) {
    const int s = tid + q * NT, k2 = s / H, lc = s % H;
    const float2* p = sm + lc * S + N1 * k2;
    float am[MODE == 0 ? N1 : 1];
    if constexpr (MODE == 0) {
#pragma unroll
      for (int i = 0; i < N1; ++i) am[i] = __ldg(a.amp + (size_t)t * M * M + (i + N1 * k2) * M + row0 + lc);
    }
    float2 v[N1];
#pragma unroll
    for (int i = 0; i < N1; ++i) v[i] = p[i];
    Dft<N1, false>::run(v);
#pragma unroll
    for (int i = 0; i < N1; ++i) {
      const size_t nat = (size_t)t * M * M + (k2 + N2 * i) * M + row0 + lc;
      if constexpr (MODE == 0) {
        const float dm = sqrtf(cabs2(v[i])) - am[i];
        acc = fmaf(dm, dm, acc);
      } else if constexpr (MODE == 1) {
        a.out_intensity[nat] = cabs2(v[i]);
      } else {
        a.out[nat] = MODE == 3 ? cconj(v[i]) : v[i];
      }
    }
  }
  if constexpr (MODE == 0) {
    const double w = warp_sum_exact(acc);
    if ((tid & 31) == 0) redd[tid >> 5] = w;
    __syncthreads();
    double part = 0.0;
    if (tid == 0)
      for (int i = 0; i < NT / 32; ++i) part += redd[i];
    if constexpr (C > 1) {
      // only rank 0 needs the parts; no CTA touches another's memory after this barrier
      if (tid == 0) *tile_rank<C>(cl, rank, &xd[rank], 0) = part;
      cl.sync();
    } else if (tid == 0) {
      xd[0] = part;
    }
    if (rank == 0 && tid == 0) {
      double tot = 0.0;
#pragma unroll
      for (int d = 0; d < C; ++d) tot += xd[d];
      a.partial[t] = tot * (0.5 / (double)(M * M));
    }
  }
}

// ---------------------------------------------------------------------------
// Wirtinger gradient of the exit-wave misfit per position (Sec. 2.1), with the
// revised exit wave recomputed: forward FFT, modulus replacement, inverse FFT,
// then gz = conj(Q) (psi - R), gq = conj(z_k) (psi - R) on the patch.
// One slab per CTA, a_k by cp.async beside it, z_k read again from L2 at the
// end: 32 warps per SM (as for the forward kernels and the step at m = 256).
// Cluster i takes positions i, i + grid, ... of the chunk, adds their probe
// gradients up in its own slot and fetches the next position's a_k while it
// finishes the current one.  With one CTA per position the grid is one wave
// (one L2-resident probe gradient per CTA instead of one per position to write
// and read back); clusters of 8 are launched one per position, since the
// hardware then fills each SM as it frees up (1600 positions at m = 256: 1.65
// ms, one wave 1.75).  us per call before -> after, with the sums: 900 positions
// at m = 128 244 -> 173, 1444 at m = 64 125 -> 68, 4096 at m = 32 133 -> 64.
template <int M, int C = WaveCluster<M>::value>
__global__ void __launch_bounds__(WaveTile<M, C>::NT, WaveTile<M, C>::MIN_CTAS) k_gradc(const GradArgs a) {
  using TL = WaveTile<M, C>;
  constexpr int NT = TL::NT, H = TL::H, S = TL::S, N1 = TL::N1, SLOTS = TL::SLOTS, PER = TL::PER;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = C == 1 ? 0 : (int)cl.block_rank();
  extern __shared__ __align__(16) float2 sm[];
  float* ampbuf = reinterpret_cast<float*>(sm + TL::slab);  // a_k on my storage columns, [M][H]
  __shared__ double xd[C];
  __shared__ float redf[(NT + 31) / 32];
  const int tid = threadIdx.x;
  const int slot = blockIdx.x / C, slots = gridDim.x / C;
  const int row0 = rank * H;
  auto fetch_amp = [&](int kb) {
    const float* amp = a.amp + (size_t)(a.first + kb) * M * M + row0;
#pragma unroll
    for (int i = tid; i < M * H / 4; i += NT)
      cp_async16(ampbuf + 4 * i, amp + (i / (H / 4)) * M + 4 * (i % (H / 4)));
    cp_async_commit();
  };
  fetch_amp(slot);
  pdl_trigger();
  for (int kb = slot; kb < a.b; kb += slots) {
  const int k = a.first + kb;
  const int o_r = a.pos[2 * k], o_c = a.pos[2 * k + 1];
  // a thread's pixels: one column, RPT rows apart
  constexpr int UL = PER < 8 ? PER : 8, RPT = NT / M;
  static_assert(NT % M == 0, "a thread's pixels share one column");
  const ObjectColumn zc(a.object, a.n_rows, a.n_cols, o_r + row0 + tid / M, o_c + tid % M);
  const float2* q = a.probe + row0 * M + tid;
  float2* mine = sm + (tid / M) * S + tid % M;
#pragma unroll (UL)
  for (int t = 0; t < PER; ++t) mine[t * RPT * S] = cmul(q[t * NT], zc.at(t * RPT));
  __syncthreads();
  gpass_a_fwd<M, H, S, 1, NT>(sm, tid);
  cp_async_wait_all();  // a_k; the barriers below show it to the whole CTA
  __syncthreads();
  row_pass_b_to_cols<TL>(cl, rank, sm, sm, tid);
  tile_sync<C>(cl);
  gpass_a_fwd<M, H, S, 1, NT>(sm, tid);
  __syncthreads();
  const float inv_m2 = 1.f / (float)(M * M);
  float acc = 0.f;
#pragma unroll
  for (int t = 0; t < SLOTS; ++t) {
    const int s = tid + t * NT, k2 = s / H, lc = s % H;
    float2* p = sm + lc * S + N1 * k2;
    float2 v[N1];
#pragma unroll
    for (int i = 0; i < N1; ++i) v[i] = p[i];
    Dft<N1, false>::run(v);
#pragma unroll
    for (int i = 0; i < N1; ++i) {
      const float am = ampbuf[(i + N1 * k2) * H + lc];
      const float p2 = cabs2(v[i]);
      if (p2 > 0.f) {
        const float inv = rsqrtf(p2);
        const float dm = fmaf(p2, inv, -am);
        acc = fmaf(dm, dm, acc);
        v[i] = cscale(v[i], am * inv * inv_m2);
      } else {
        acc = fmaf(am, am, acc);
        v[i] = make_float2(am * inv_m2, 0.f);
      }
    }
    Dft<N1, true>::run(v);
#pragma unroll
    for (int i = 0; i < N1; ++i) p[i] = v[i];
  }
  // per-warp misfit partials; the barrier also orders the pass before the next one
  warp_partial_sum(acc, redf);
  __syncthreads();
  // rank 0 collects the parts (every CTA has started: the row pass waited for them all)
  if (tid == 0) *tile_rank<C>(cl, rank, &xd[rank], 0) = partials_sum<NT>(redf);
  col_pass_a_inv_to_rows<TL>(cl, rank, sm, sm, tid);
  tile_sync<C>(cl);
  if (kb + slots < a.b) fetch_amp(kb + slots);  // ampbuf has been read
  gpass_b<M, H, S, 1, NT, true>(sm, tid);
  __syncthreads();
  gpass_a_inv<M, H, S, 1, NT>(sm, tid);
  __syncthreads();
  float2* gz = a.gz + (size_t)kb * M * M + row0 * M + tid;
  float2* gq = a.gq + (size_t)slot * M * M + row0 * M + tid;
  const bool more = k != slot;  // this slot holds a sum already (of this launch or an earlier chunk's)
  // patch gradients; the loads of UG pixels of a thread are issued together
  constexpr int UG = PER < 4 ? PER : 4;
#pragma unroll 1
  for (int t0 = 0; t0 < PER; t0 += UG) {
    float2 qv[UG], zv[UG];
#pragma unroll
    for (int u = 0; u < UG; ++u) {
      qv[u] = __ldg(q + (t0 + u) * NT);
      zv[u] = zc.at((t0 + u) * RPT);
    }
#pragma unroll
    for (int u = 0; u < UG; ++u) {
      const float2 e = csub(cmul(qv[u], zv[u]), mine[(t0 + u) * RPT * S]);
      gz[(t0 + u) * NT] = cconjmul(qv[u], e);
      // one thread adds to each address, so the order of the sum is fixed
      if (more)
        atomicAdd(gq + (t0 + u) * NT, cconjmul(zv[u], e));
      else
        gq[(t0 + u) * NT] = cconjmul(zv[u], e);
    }
  }
  if (rank == 0 && tid == 0) {
    double tot = 0.0;
#pragma unroll
    for (int d = 0; d < C; ++d) tot += xd[d];
    a.phi[kb] = tot * (0.5 / (double)(M * M));
  }
  __syncthreads();  // the slab has been read before the next position's gather
  }
}

// Object gradient sum_k P_k^T gz_k over tiles of 8 PX x 32 pixels (optionally
// added to the existing values: later chunks of positions) and probe gradient
// sum of the slots' gq, each in a fixed order (deterministic).  Bound by
// the loads: a thread keeps those of U patches at PX pixels in flight, and
// the positions that overlap a tile are listed kGradList at a time, so any number
// of positions takes the same shared memory.  PX = 2, U = 4; objects with fewer
// than kGradSmallTiles such tiles (two per SM) take PX = 1, U = 8, or they would
// leave SMs idle (us per call of 1444 positions: object 192^2 and m = 64 142 / 113,
// 320^2 and m = 128 443 / 371).  Each tile reads all positions, so more tiles
// cost more where many positions miss them: 512^2, 4096 positions, m = 32 51 / 58.
constexpr int kGradList = 512, kGradSmallTiles = 304, kGradTileW = 32, kGradTileH = kApplyThreads / 32;
template <int PX, int U>
__global__ void __launch_bounds__(kApplyThreads) k_grad_reduce(const GradReduceArgs a) {
  constexpr int WARPS = kApplyThreads / 32, PW = kGradList / WARPS, ROUNDS = PW / 32, PP = kApplyProbePx / 32;
  constexpr int TILE_H = PX * WARPS;
  static_assert(WARPS == kApplyProbeGroups && (PX == 1 || PX == 2), "one or two tile rows per warp");
  __shared__ int3 list[kGradList];
  __shared__ int count[WARPS];
  __shared__ float2 part_s[kApplyProbeGroups][kApplyProbePx];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n_tiles = a.tiles_x * a.tiles_y;
  const int m = a.m;
  const size_t mm = (size_t)m * m;
  pdl_trigger();
  if ((int)blockIdx.x < n_tiles) {
    if (!a.grad_object) return;
    const int r0 = (int)(blockIdx.x / a.tiles_x) * TILE_H, c0 = (int)(blockIdx.x % a.tiles_x) * kGradTileW;
    bool waited = false;
    const int row = r0 + warp, col = c0 + lane;  // pixels (row + h WARPS, col)
    float2 g[PX];
#pragma unroll
    for (int h = 0; h < PX; ++h) g[h] = czero();
    for (int k0 = 0; k0 < a.b; k0 += kGradList) {
      // ordered compaction: warp w lists the w-th run of these positions
      int3 p[ROUNDS];
      unsigned mask[ROUNDS];
      int mine = 0;
#pragma unroll
      for (int i = 0; i < ROUNDS; ++i) {
        const int kb = k0 + warp * PW + i * 32 + lane;
        bool hit = false;
        if (kb < a.b) {
          p[i] = make_int3(kb, a.pos[2 * (a.first + kb)], a.pos[2 * (a.first + kb) + 1]);
          hit = p[i].y < r0 + TILE_H && p[i].y + m > r0 && p[i].z < c0 + kGradTileW && p[i].z + m > c0;
        }
        mask[i] = __ballot_sync(0xffffffffu, hit);
        mine += __popc(mask[i]);
      }
      __syncthreads();  // the previous list has been walked
      if (lane == 0) count[warp] = mine;
      __syncthreads();
      int at = 0, total = 0;
#pragma unroll
      for (int w = 0; w < WARPS; ++w) {
        if (w < warp) at += count[w];
        total += count[w];
      }
#pragma unroll
      for (int i = 0; i < ROUNDS; ++i) {
        if (mask[i] >> lane & 1u) list[at + __popc(mask[i] & ((1u << lane) - 1u))] = p[i];
        at += __popc(mask[i]);
      }
      __syncthreads();
      if (!waited) pdl_wait();  // the patch gradients; the first list needs the positions alone
      waited = true;
      for (int t0 = 0; t0 < total; t0 += U) {
        float2 v[U][PX];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          v[u][0] = v[u][PX - 1] = czero();
          if (t0 + u < total) {
            const int3 q = list[t0 + u];
            const int lr = row - q.y, lc = col - q.z;
            const float2* src = a.gz + (size_t)q.x * mm + lr * m + lc;
            const bool in_c = (unsigned)lc < (unsigned)m;
            if (in_c && (unsigned)lr < (unsigned)m) v[u][0] = src[0];
            if constexpr (PX > 1)
              if (in_c && (unsigned)(lr + WARPS) < (unsigned)m) v[u][1] = src[WARPS * m];
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int h = 0; h < PX; ++h) g[h] = cadd(g[h], v[u][h]);
      }
    }
    if (col >= a.n_cols) return;
#pragma unroll
    for (int h = 0; h < PX; ++h) {
      if (row + h * WARPS >= a.n_rows) continue;
      const size_t gi = (size_t)(row + h * WARPS) * a.n_cols + col;
      a.grad_object[gi] = a.accumulate ? cadd(a.grad_object[gi], g[h]) : g[h];
    }
  } else {
    if (!a.grad_probe) return;
    pdl_wait();
    const int p0 = (blockIdx.x - n_tiles) * kApplyProbePx + lane;  // pixels p0 + 32 h; warp w sums slots w, w + 8, ...
    float2 s[PP];
#pragma unroll
    for (int h = 0; h < PP; ++h) s[h] = czero();
    for (int k0 = warp; k0 < a.slots; k0 += 4 * kApplyProbeGroups) {
      float2 v[4][PP];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int h = 0; h < PP; ++h) {
          const int k = k0 + u * kApplyProbeGroups;
          v[u][h] = k < a.slots && p0 + 32 * h < (int)mm ? a.gq[(size_t)k * mm + p0 + 32 * h] : czero();
        }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int h = 0; h < PP; ++h) s[h] = cadd(s[h], v[u][h]);
    }
#pragma unroll
    for (int h = 0; h < PP; ++h) part_s[warp][lane + 32 * h] = s[h];
    __syncthreads();
    const int p = (blockIdx.x - n_tiles) * kApplyProbePx + tid;
    if (tid >= kApplyProbePx || p >= (int)mm) return;
    float2 tot = part_s[0][tid];
#pragma unroll
    for (int i = 1; i < kApplyProbeGroups; ++i) tot = cadd(tot, part_s[i][tid]);
    a.grad_probe[p] = tot;
  }
}

// ---------------------------------------------------------------------------
// a8 + a9: deterministic combine.  Blocks [0, tiles) own object tiles of
// kApplyTile x kApplyTileW pixels (kApplyPx pixels per thread, kApplyTile
// apart in the row); the remaining blocks own kApplyProbePx probe pixels each
// (kApplyProbePx / 32 per lane), with 8 thread groups summing disjoint
// position subsets that are then added in a fixed order.  Each thread issues
// the loads of all its pixels together, and the grid of the bench-sized
// object and probe is resident at once after the step.  The new probe's
// max|Q|^2 goes to a.mq_next for the next prep.
#ifndef EMG_APPLY_MIN_BLOCKS
#define EMG_APPLY_MIN_BLOCKS 4
#endif
#ifndef EMG_APPLY_CHUNK
#define EMG_APPLY_CHUNK 4
#endif
constexpr int kApplyChunk = EMG_APPLY_CHUNK;  // covering patches whose loads a thread issues together
__global__ void __launch_bounds__(kApplyThreads, EMG_APPLY_MIN_BLOCKS) k_apply(const ApplyArgs a) {
  constexpr int PX = kApplyPx, PP = kApplyProbePx / 32;
  extern __shared__ int list[];  // [b][3] = (kb, row, col) of patches overlapping the tile
  __shared__ int warp_count[kApplyThreads / 32];
  __shared__ int total;
  __shared__ float2 part_s[kApplyProbeGroups][kApplyProbePx];
  __shared__ int part_n[kApplyProbeGroups][kApplyProbePx];
  const int tid = threadIdx.x;
  const int n_tiles = a.tiles_x * a.tiles_y;
  const int m = a.m;
  const size_t mm = (size_t)m * m;
  pdl_trigger();
  if ((int)blockIdx.x < n_tiles && a.s_num) {
    // atomic scatter: the step kernel has accumulated this tile's sums; finalise and reset them
    const int ty = blockIdx.x / a.tiles_x, tx = blockIdx.x % a.tiles_x;
    const int row = ty * kApplyTile + tid / kApplyTile;
    if (row >= a.n_rows) return;
    pdl_wait();
#pragma unroll
    for (int h = 0; h < PX; ++h) {
      const int col = tx * kApplyTileW + tid % kApplyTile + h * kApplyTile;
      if (col >= a.n_cols) continue;
      const size_t gi = (size_t)row * a.n_cols + col;
      if (a.combine == 0) {
        const float den = a.s_den[gi];
        if (den > 0.f) {
          a.object[gi] = cscale(a.s_num[gi], 1.f / den);
          a.s_num[gi] = czero();
          a.s_den[gi] = 0.f;
        }
      } else {
        const float2 dz = a.s_num[gi];
        if (dz.x != 0.f || dz.y != 0.f) {
          a.object[gi] = cadd(a.object[gi], dz);
          a.s_num[gi] = czero();
        }
      }
    }
  } else if ((int)blockIdx.x < n_tiles) {
    const int ty = blockIdx.x / a.tiles_x, tx = blockIdx.x % a.tiles_x;
    const int r0 = ty * kApplyTile, c0 = tx * kApplyTileW;
    if (tid == 0) total = 0;
    __syncthreads();
    // ordered compaction of the minibatch patches that overlap this tile
    for (int base = 0; base < a.b; base += kApplyThreads) {
      const int kb = base + tid;
      int pr = 0, pc = 0;
      bool hit = false;
      if (kb < a.b) {
        int k = a.order[kb];
        if (!EMG_INB(k, a.n_pos, kBcApplyOrder)) k = 0;
        pr = a.pos[2 * k];
        pc = a.pos[2 * k + 1];
        hit = pr < r0 + kApplyTile && pr + m > r0 && pc < c0 + kApplyTileW && pc + m > c0;
      }
      const unsigned mask = __ballot_sync(0xffffffffu, hit);
      const int lane = tid & 31, warp = tid >> 5;
      if (lane == 0) warp_count[warp] = __popc(mask);
      __syncthreads();
      int off = total;
      for (int w = 0; w < warp; ++w) off += warp_count[w];
      if (hit) {
        const int slot = off + __popc(mask & ((1u << lane) - 1u));
        list[3 * slot] = kb;
        list[3 * slot + 1] = pr;
        list[3 * slot + 2] = pc;
      }
      __syncthreads();
      if (tid == 0) {
        int t = total;
        for (int w = 0; w < kApplyThreads / 32; ++w) t += warp_count[w];
        total = t;
      }
      __syncthreads();
    }
    const int cnt = total;
    const int row = r0 + tid / kApplyTile, col0 = c0 + tid % kApplyTile;
    if (cnt == 0 || row >= a.n_rows || col0 >= a.n_cols) return;
    pdl_wait();  // patches z~_k and weights come from the step and prep kernels
    float2 num[PX];
    float den[PX];
    bool covered[PX];
#pragma unroll
    for (int h = 0; h < PX; ++h) {
      num[h] = czero();
      den[h] = 0.f;
      covered[h] = false;
    }
    // patches in minibatch order; loads of kApplyChunk patches at all pixels are issued together
    for (int t0 = 0; t0 < cnt; t0 += kApplyChunk) {
      float2 v[PX][kApplyChunk];
      float w[PX][kApplyChunk];
      bool in[PX][kApplyChunk];
#pragma unroll
      for (int u = 0; u < kApplyChunk; ++u) {
        const int t = t0 + u;
#pragma unroll
        for (int h = 0; h < PX; ++h) in[h][u] = false;
        if (t < cnt) {
          const int kb = list[3 * t], lr = row - list[3 * t + 1], lc = col0 - list[3 * t + 2];
          const bool ok = (unsigned)lr < (unsigned)m && EMG_INB(kb, a.b, kBcApplyPatch);
          // all pixels from one base address: pixel h is h kApplyTile columns on
          const float2* zrow = a.zt + (size_t)kb * mm + lr * m + lc;
          const float* wrow = a.wq + lr * m + lc;
#pragma unroll
          for (int h = 0; h < PX; ++h) {
            in[h][u] = ok && (unsigned)(lc + h * kApplyTile) < (unsigned)m && col0 + h * kApplyTile < a.n_cols;
            if (in[h][u]) {
              v[h][u] = zrow[h * kApplyTile];
              w[h][u] = a.combine == 0 ? wrow[h * kApplyTile] : 1.f;
            }
          }
        }
      }
#pragma unroll
      for (int h = 0; h < PX; ++h)
#pragma unroll
        for (int u = 0; u < kApplyChunk; ++u) {
          if (in[h][u]) {
            covered[h] = true;
            if (a.combine == 0) {
              num[h] = make_float2(fmaf(w[h][u], v[h][u].x, num[h].x), fmaf(w[h][u], v[h][u].y, num[h].y));
            } else {
              num[h] = cadd(num[h], v[h][u]);
            }
            den[h] += w[h][u];
          }
        }
    }
#pragma unroll
    for (int h = 0; h < PX; ++h) {
      if (!covered[h]) continue;
      const size_t gi = (size_t)row * a.n_cols + col0 + h * kApplyTile;
      if (!EMG_INB(gi, (size_t)a.n_rows * a.n_cols, kBcApplyObject)) continue;
      if (a.combine == 0) {
        a.object[gi] = safe_cdiv(num[h], den[h]);
      } else {
        const float2 z = a.object[gi];
        a.object[gi] = cadd(z, csub(num[h], cscale(z, den[h])));
      }
    }
  } else {
    pdl_wait();  // probes Q~_k come from the step kernel
    const int lane = tid & 31, g = tid >> 5;
    const int p0 = (blockIdx.x - n_tiles) * kApplyProbePx + lane;
    float2 s[PP];
#pragma unroll
    for (int h = 0; h < PP; ++h) s[h] = czero();
    int cnt = 0;
    if (p0 < (int)mm) {
      for (int kb0 = g; kb0 < a.b; kb0 += 4 * kApplyProbeGroups) {
        float2 v[PP][4];
        float mu[4];
        // mu_k and Q~_k are loaded together; slots with mu_k = 0 are skipped when summing
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int kb = kb0 + u * kApplyProbeGroups;
          mu[u] = 0.f;
          if (kb < a.b) {
            mu[u] = a.mu[kb];
            const float2* qrow = a.qt + (size_t)kb * mm + p0;
#pragma unroll
            for (int h = 0; h < PP; ++h)
              if (p0 + 32 * h < (int)mm) v[h][u] = qrow[32 * h];
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (mu[u] > 0.f) {
#pragma unroll
            for (int h = 0; h < PP; ++h)
              if (p0 + 32 * h < (int)mm) s[h] = cadd(s[h], v[h][u]);
            ++cnt;
          }
        }
      }
    }
#pragma unroll
    for (int h = 0; h < PP; ++h) {
      part_s[g][lane + 32 * h] = s[h];
      part_n[g][lane + 32 * h] = cnt;
    }
    __syncthreads();
    if (tid >= kApplyProbePx) return;
    const int p = (blockIdx.x - n_tiles) * kApplyProbePx + tid;
    float a2 = 0.f;
    if (p < (int)mm) {
      float2 tot = part_s[0][tid];
      int n = part_n[0][tid];
#pragma unroll
      for (int i = 1; i < kApplyProbeGroups; ++i) {
        tot = cadd(tot, part_s[i][tid]);
        n += part_n[i][tid];
      }
      float2 q = a.probe[p];
      if (n > 0) {
        q = (a.combine == 0) ? cscale(tot, 1.f / (float)n) : cadd(q, csub(tot, cscale(q, (float)n)));
        a.probe[p] = q;
      }
      a2 = cabs2(q);
    }
    if (a.mq_next) warp_atomic_max(a.mq_next, a2);
  }
}

// ---------------------------------------------------------------------------
// Deterministic single-block sum: out = scale * sum x[0..n).
constexpr int kSumThreads = 256;  // 1024 threads: 13.8 us for 1444 values, most of it the FP64 trees
__global__ void __launch_bounds__(kSumThreads) k_sum(const double* __restrict__ x, int n,
                                                     double scale, double* __restrict__ out) {
  __shared__ double redd[kSumThreads / 32];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += kSumThreads) s += x[i];
  s = block_sum<kSumThreads>(s, redd);
  if (threadIdx.x == 0) *out = s * scale;
}

// dp_avg probe scaling (Sec. 4.1): partial sums of a^2 = max(d, 0).
constexpr int kNormThreads = 256;
__global__ void __launch_bounds__(kNormThreads) k_sum_sq(const float* __restrict__ amp, size_t n,
                                                         double* __restrict__ partial) {
  __shared__ double redd[kNormThreads / 32];
  double s = 0.0;
  for (size_t i = blockIdx.x * (size_t)kNormThreads + threadIdx.x; i < n;
       i += (size_t)gridDim.x * kNormThreads) {
    const float v = amp[i];
    s += (double)(v * v);
  }
  s = block_sum<kNormThreads>(s, redd);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

constexpr int kScaleThreads = 1024;
__global__ void __launch_bounds__(kScaleThreads) k_scale_probe(const double* __restrict__ partial,
                                                             int n_partial, int m, int n_pos,
                                                             float2* __restrict__ probe) {
  __shared__ double redd[kScaleThreads / 32];
  double s = 0.0;
  for (int i = threadIdx.x; i < n_partial; i += kScaleThreads) s += partial[i];
  const double sum_d = block_sum<kScaleThreads>(s, redd);
  double q2 = 0.0;
  for (int p = threadIdx.x; p < m * m; p += kScaleThreads) q2 += (double)cabs2(probe[p]);
  const double norm2 = block_sum<kScaleThreads>(q2, redd);
  const double dp_avg = sqrt(sum_d / (double)n_pos) / (double)m;
  const float scale = norm2 > 0.0 ? (float)(dp_avg / sqrt(norm2)) : 0.f;
  for (int p = threadIdx.x; p < m * m; p += kScaleThreads) probe[p] = cscale(probe[p], scale);
}

#define EMG_DISPATCH_M(m, CALL)        \
  switch (m) {                         \
    case 16: { constexpr int M = 16; return CALL; }   \
    case 32: { constexpr int M = 32; return CALL; }   \
    case 64: { constexpr int M = 64; return CALL; }   \
    case 128: { constexpr int M = 128; return CALL; } \
    case 256: { constexpr int M = 256; return CALL; } \
    default: return cudaErrorInvalidValue;            \
  }

}  // namespace

// Dynamic shared memory per CTA; 227 KB minus room for the kernels' static reductions.
// Launch with programmatic stream serialisation (see pdl_wait / pdl_trigger).
template <typename Kernel, typename... Args>
cudaError_t launch_pdl(Kernel kernel, dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

int step_smem_limit() { return 227 * 1024 - 1024; }

size_t step_smem_bytes(int m, int levels) {
  switch (m) {
    case 16: return step_smem_elems<16>(levels) * sizeof(float2);
    case 32: return step_smem_elems<32>(levels) * sizeof(float2);
    case 64: return step_smem_elems<64>(levels) * sizeof(float2);
    case 128: return step_smem_elems<128>(levels) * sizeof(float2);
    default: return 0;
  }
}

cudaError_t set_cluster_attrs();

cudaError_t upload_twiddles() {
  float2 h[256];
  for (int t = 0; t < 256; ++t) {
    const double ang = -2.0 * M_PI * (double)t / 256.0;
    double c = cos(ang), s = sin(ang);
    if (fabs(c) < 1e-15) c = 0.0;
    if (fabs(s) < 1e-15) s = 0.0;
    h[t] = make_float2((float)c, (float)s);
  }
  cudaError_t e = cudaMemcpyToSymbol(c_twiddle, h, sizeof(h));
  if (e != cudaSuccess) return e;
  float2 st[16 + 32 + 64 + 128];
  auto fill = [&](int m, int n1, int n2) {
    for (int j = 0; j < n1; ++j)
      for (int k = 0; k < n2; ++k) st[m - 16 + j * n2 + k] = h[(j * k) % m * (256 / m)];
  };
  fill(16, FftPlan<16>::N1, FftPlan<16>::N2);
  fill(32, FftPlan<32>::N1, FftPlan<32>::N2);
  fill(64, FftPlan<64>::N1, FftPlan<64>::N2);
  fill(128, FftPlan<128>::N1, FftPlan<128>::N2);
  e = cudaMemcpyToSymbol(c_stage, st, sizeof(st));
  if (e != cudaSuccess) return e;
  if ((e = set_cluster_attrs()) != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_apply, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_prep_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPrepTileSmemMax);
  return e;
}

cudaError_t launch_amp_prep(const float* d, float* amp, int m, int n_pos, cudaStream_t s) {
  const size_t rows = (size_t)n_pos * m;
  int blocks = (int)((rows + 7) / 8);
  if (blocks > 152 * 8) blocks = 152 * 8;
  if (blocks == 0) return cudaSuccess;
  switch (m) {
    case 16: k_amp_prep<16><<<blocks, 256, 0, s>>>(d, amp, n_pos); break;
    case 32: k_amp_prep<32><<<blocks, 256, 0, s>>>(d, amp, n_pos); break;
    case 64: k_amp_prep<64><<<blocks, 256, 0, s>>>(d, amp, n_pos); break;
    case 128: k_amp_prep<128><<<blocks, 256, 0, s>>>(d, amp, n_pos); break;
    case 256: k_amp_prep<256><<<blocks, 256, 0, s>>>(d, amp, n_pos); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// Shared memory each gather block reserves in all (its row buffer plus unused
// dynamic shared memory, within the 48 KB a launch may ask for without opting
// in).  At the bench size a block that large does not fit beside two step
// CTAs, so the gathers run on the SMs the step leaves free instead of slowing
// its CTAs: end to end 1.57M -> 1.62M positions/s (20 KB per block gave 1.44M).
#ifndef EMG_GATHER_BLOCK_SMEM
#define EMG_GATHER_BLOCK_SMEM (46 * 1024)
#endif
cudaError_t launch_amp_gather(const float* d, const int32_t* idx, int b, float* amp, int m, cudaStream_t s) {
  const int groups = b * (m / kGatherRows);
  int blocks = (groups + kGatherWarps - 1) / kGatherWarps;
  if (blocks > kGatherBlocks) blocks = kGatherBlocks;
  if (blocks == 0) return cudaSuccess;
  const dim3 th(kGatherWarps * 32);
  const size_t rows_bytes = (size_t)kGatherWarps * kGatherRows * m * sizeof(float);
  const size_t pad = rows_bytes < EMG_GATHER_BLOCK_SMEM ? EMG_GATHER_BLOCK_SMEM - rows_bytes : 0;
  switch (m) {
    case 16: k_amp_gather<16><<<blocks, th, pad, s>>>(d, idx, b, amp); break;
    case 32: k_amp_gather<32><<<blocks, th, pad, s>>>(d, idx, b, amp); break;
    case 64: k_amp_gather<64><<<blocks, th, pad, s>>>(d, idx, b, amp); break;
    case 128: k_amp_gather<128><<<blocks, th, pad, s>>>(d, idx, b, amp); break;
    case 256: k_amp_gather<256><<<blocks, th, pad, s>>>(d, idx, b, amp); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

#ifndef EMG_PREP_TILE
#define EMG_PREP_TILE 8
#endif
bool prep_tiled_config(PrepArgs& a) {
  int tile = EMG_PREP_TILE;
  while (tile < (1 << (a.levels - 1))) tile *= 2;
  if (tile > a.m) tile = a.m;
  a.tile = tile;
  a.halo = (a.prolong == 1) ? (1 << (a.levels - 1)) : 0;
  if ((tile >> (a.levels - 1)) < 1) return false;
  return prep_tile_smem(a) <= kPrepTileSmemMax;
}

template <int M, int C>
constexpr size_t stepc_smem_bytes() {
  return StepTile<M, C>::smem_elems * sizeof(float2);
}

// Clusters of the step kernel that can be resident at once (CTAs per SM from
// the occupancy calculator x SMs / cluster size), or 0 if unknown.
template <int M, int C>
int stepc_resident_clusters() {
  int per_sm = 0, dev = 0, sms = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_stepc<M, C>, StepTile<M, C>::NT,
                                                    stepc_smem_bytes<M, C>()) != cudaSuccess ||
      cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return per_sm * sms / C;
}

int step_resident_clusters(int m, int cluster) {
  switch (m * 16 + cluster) {
    case 16 * 16 + 1: return stepc_resident_clusters<16, 1>();
    case 32 * 16 + 1: return stepc_resident_clusters<32, 1>();
    case 16 * 16 + 2: return stepc_resident_clusters<16, 2>();
    case 32 * 16 + 2: return stepc_resident_clusters<32, 2>();
    case 64 * 16 + 2: return stepc_resident_clusters<64, 2>();
    case 64 * 16 + 4: return stepc_resident_clusters<64, 4>();
    case 128 * 16 + 2: return stepc_resident_clusters<128, 2>();
    case 128 * 16 + 4: return stepc_resident_clusters<128, 4>();
    case 128 * 16 + 8: return stepc_resident_clusters<128, 8>();
    case 256 * 16 + 8: return stepc_resident_clusters<256, 8>();
    default: return 0;
  }
}

int fused_prep_tiles(PrepArgs& a, int m, int cluster) {
  size_t smem = 0;
  switch (m * 16 + cluster) {
    case 16 * 16 + 1: smem = stepc_smem_bytes<16, 1>(); break;
    case 32 * 16 + 1: smem = stepc_smem_bytes<32, 1>(); break;
    case 16 * 16 + 2: smem = stepc_smem_bytes<16, 2>(); break;
    case 32 * 16 + 2: smem = stepc_smem_bytes<32, 2>(); break;
    case 64 * 16 + 2: smem = stepc_smem_bytes<64, 2>(); break;
    case 64 * 16 + 4: smem = stepc_smem_bytes<64, 4>(); break;
    case 128 * 16 + 2: smem = stepc_smem_bytes<128, 2>(); break;
    case 128 * 16 + 4: smem = stepc_smem_bytes<128, 4>(); break;
    case 128 * 16 + 8: smem = stepc_smem_bytes<128, 8>(); break;
    case 256 * 16 + 8: smem = stepc_smem_bytes<256, 8>(); break;
    default: return 0;
  }
  // a quarter of the side, so that a small probe's prep is shared by as many
  // CTAs and ends before the transforms do (us per minibatch of 64 with three
  // levels, tiles of 32 against these: m = 64 19.8 / 17.7, m = 32 18.0 / 14.6)
  int tile = m / 4 < 8 ? 8 : m / 4 > 32 ? 32 : m / 4;
  while (tile < (1 << (a.levels - 1))) tile *= 2;
  if (tile > m) tile = m;
  a.tile = tile;
  a.halo = (a.prolong == 1) ? (1 << (a.levels - 1)) : 0;
  if ((tile >> (a.levels - 1)) < 1 || prep_tile_smem(a) > smem) return 0;
  return (m / tile) * (m / tile);
}

cudaError_t launch_prep(const PrepArgs& a, bool overlap, cudaStream_t s) {
  PrepArgs t = a;
  if (a.mq_read && prep_tiled_config(t)) {
    const int tiles = (t.m / t.tile) * (t.m / t.tile);
    if (overlap) {
      cudaError_t e = launch_pdl(k_prep_tile, dim3(tiles), dim3(kPrepTileThreads), prep_tile_smem(t), s, t);
      if (e != cudaSuccess) return e;
    } else {
      k_prep_tile<<<tiles, kPrepTileThreads, prep_tile_smem(t), s>>>(t);
    }
  } else {
    k_prep<<<1, kPrepThreads, 0, s>>>(a);
  }
  return cudaGetLastError();
}

// Launch of a C-CTA cluster kernel with programmatic stream serialisation.
template <typename Kernel, typename... Args>
cudaError_t launch_cluster_pdl(Kernel kernel, int cluster, dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                               Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename Kernel, typename... Args>
cudaError_t launch_cluster_plain(Kernel kernel, int cluster, dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                 Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <int NI>
cudaError_t launch_seed_t(const float2* probe, int m, unsigned* mq, unsigned* sync, int32_t* order, const int32_t* idx,
                          int b, cudaStream_t s) {
  SeedIdx<NI> pv;
  if (NI > 0) memcpy(pv.v, idx, (size_t)b * sizeof(int32_t));
  const int ctas = m <= 64 ? 1 : kSeedCtas;  // 4096 pixels are 8 loads a thread for one CTA
  const cudaError_t e = launch_cluster_pdl(k_seed<NI>, ctas, dim3(ctas), dim3(kSeedThreads), 0, s, probe, m * m, mq, sync,
                                           order, b, pv);
  return e != cudaSuccess ? e : cudaGetLastError();
}

bool seed_takes_idx(int b) { return b <= kSeedMaxIdx; }

cudaError_t launch_seed(const float2* probe, int m, unsigned* mq, unsigned* sync, int32_t* order, const int32_t* idx, int b,
                        cudaStream_t s) {
  if (!idx) return launch_seed_t<0>(probe, m, mq, sync, nullptr, nullptr, 0, s);
  if (b <= 64) return launch_seed_t<64>(probe, m, mq, sync, order, idx, b, s);
  return launch_seed_t<kSeedMaxIdx>(probe, m, mq, sync, order, idx, b, s);
}

template <int M, int MODE>
cudaError_t launch_forward_t(int count, const FwdArgs& a, cudaStream_t s) {
  using TL = WaveTile<M>;
  constexpr size_t bytes = TL::slab * sizeof(float2);
  if constexpr (TL::CTAS == 1) {
    k_forward<M, MODE><<<count, TL::NT, bytes, s>>>(a);
  } else {
    cudaError_t e = launch_cluster_plain(k_forward<M, MODE>, TL::CTAS, dim3(TL::CTAS * count), dim3(TL::NT), bytes, s, a);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

template <int M, int C = WaveCluster<M>::value>
constexpr size_t gradc_smem_elems() {
  return WaveTile<M, C>::slab + (size_t)WaveTile<M, C>::H * M / 2;
}

template <int M, int C = WaveCluster<M>::value>
cudaError_t launch_gradc_t(int slots, const GradArgs& a, cudaStream_t s) {
  using TL = WaveTile<M, C>;
  constexpr size_t bytes = gradc_smem_elems<M, C>() * sizeof(float2);
  const cudaError_t e =
      launch_cluster_plain(k_gradc<M, C>, TL::CTAS, dim3(TL::CTAS * slots), dim3(TL::NT), bytes, s, a);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename Kernel>
cudaError_t set_cluster_smem(Kernel k, size_t elems) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(elems * sizeof(float2)));
}

template <int M, int C, bool RIN = false>
cudaError_t set_stepc_attrs() {
  return set_cluster_smem(k_stepc<M, C, RIN>, StepTile<M, C>::smem_elems);
}

template <int M>
cudaError_t set_forward_attrs() {
  cudaError_t e;
  if ((e = set_cluster_smem(k_forward<M, 0>, WaveTile<M>::slab)) != cudaSuccess) return e;
  if ((e = set_cluster_smem(k_forward<M, 1>, WaveTile<M>::slab)) != cudaSuccess) return e;
  if ((e = set_cluster_smem(k_forward<M, 2>, WaveTile<M>::slab)) != cudaSuccess) return e;
  return set_cluster_smem(k_forward<M, 3>, WaveTile<M>::slab);
}

template <int M, int C = WaveCluster<M>::value>
cudaError_t set_grad_attrs() {
  return set_cluster_smem(k_gradc<M, C>, gradc_smem_elems<M, C>());
}

// Dynamic shared-memory limits of the cluster kernels (once per device).
cudaError_t set_cluster_attrs() {
  cudaError_t e;
  if ((e = set_stepc_attrs<16, 1>()) != cudaSuccess) return e;
  if ((e = set_stepc_attrs<32, 1>()) != cudaSuccess) return e;
  if ((e = set_stepc_attrs<16, 2>()) != cudaSuccess) return e;
  if ((e = set_stepc_attrs<32, 2>()) != cudaSuccess) return e;
  if ((e = set_stepc_attrs<64, 2>()) != cudaSuccess) return e;
  if ((e = set_stepc_attrs<64, 4>()) != cudaSuccess) return e;
  if ((e = set_stepc_attrs<128, 2>()) != cudaSuccess) return e;
  if ((e = set_stepc_attrs<128, 4>()) != cudaSuccess) return e;
  if ((e = set_stepc_attrs<128, 8>()) != cudaSuccess) return e;
  if ((e = set_stepc_attrs<256, 8>()) != cudaSuccess) return e;
  if ((e = set_stepc_attrs<128, 2, true>()) != cudaSuccess) return e;
  if ((e = set_stepc_attrs<128, 4, true>()) != cudaSuccess) return e;
  if ((e = set_stepc_attrs<128, 8, true>()) != cudaSuccess) return e;
  if ((e = set_stepc_attrs<256, 8, true>()) != cudaSuccess) return e;
  if ((e = set_forward_attrs<16>()) != cudaSuccess) return e;
  if ((e = set_forward_attrs<32>()) != cudaSuccess) return e;
  if ((e = set_forward_attrs<64>()) != cudaSuccess) return e;
  if ((e = set_forward_attrs<128>()) != cudaSuccess) return e;
  if ((e = set_forward_attrs<256>()) != cudaSuccess) return e;
  if ((e = set_grad_attrs<16>()) != cudaSuccess) return e;
  if ((e = set_grad_attrs<32>()) != cudaSuccess) return e;
  if ((e = set_grad_attrs<64>()) != cudaSuccess) return e;
  if ((e = set_grad_attrs<128>()) != cudaSuccess) return e;
  if ((e = set_grad_attrs<128, 2>()) != cudaSuccess) return e;
  if ((e = set_grad_attrs<256>()) != cudaSuccess) return e;
  return cudaSuccess;
}

template <int M, int C>
cudaError_t launch_stepc_t(int b, const StepArgs& a, bool overlap, cudaStream_t s) {
  using TL = StepTile<M, C>;
  const dim3 grid(C * (b + a.prep_clusters)), block(TL::NT);
  constexpr size_t bytes = TL::smem_elems * sizeof(float2);
  cudaError_t e = overlap ? launch_cluster_pdl(k_stepc<M, C>, C, grid, block, bytes, s, a)
                          : launch_cluster_plain(k_stepc<M, C>, C, grid, block, bytes, s, a);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

template <int M, int C>
cudaError_t launch_stepc_rin_t(int b, const StepArgs& a, cudaStream_t s) {
  using TL = StepTile<M, C>;
  cudaError_t e = launch_cluster_pdl(k_stepc<M, C, true>, C, dim3(C * b), dim3(TL::NT),
                                     TL::smem_elems * sizeof(float2), s, a);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

cudaError_t launch_step_rin(int m, int b, const StepArgs& a, cudaStream_t s) {
  switch (m * 16 + a.cluster) {
    case 128 * 16 + 2: return launch_stepc_rin_t<128, 2>(b, a, s);
    case 128 * 16 + 4: return launch_stepc_rin_t<128, 4>(b, a, s);
    case 128 * 16 + 8: return launch_stepc_rin_t<128, 8>(b, a, s);
    case 256 * 16 + 8: return launch_stepc_rin_t<256, 8>(b, a, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_step(int m, int b, const StepArgs& a, bool overlap, cudaStream_t s) {
  switch (m * 16 + a.cluster) {
    case 16 * 16 + 1: return launch_stepc_t<16, 1>(b, a, overlap, s);
    case 16 * 16 + 2: return launch_stepc_t<16, 2>(b, a, overlap, s);
    case 32 * 16 + 1: return launch_stepc_t<32, 1>(b, a, overlap, s);
    case 32 * 16 + 2: return launch_stepc_t<32, 2>(b, a, overlap, s);
    case 64 * 16 + 2: return launch_stepc_t<64, 2>(b, a, overlap, s);
    case 64 * 16 + 4: return launch_stepc_t<64, 4>(b, a, overlap, s);
    case 128 * 16 + 2: return launch_stepc_t<128, 2>(b, a, overlap, s);
    case 128 * 16 + 4: return launch_stepc_t<128, 4>(b, a, overlap, s);
    case 128 * 16 + 8: return launch_stepc_t<128, 8>(b, a, overlap, s);
    case 256 * 16 + 8: return launch_stepc_t<256, 8>(b, a, overlap, s);
    default: return cudaErrorInvalidValue;
  }
}

// CTAs per position by default: 4 for m = 128 where every CTA keeps a row at
// the coarsest level (measured faster than 2), else the one choice built.
int default_cluster(int m, int levels) {
  if (m <= 32) return 1;
  if (m == 256) return 8;
  if (m == 128 && step_supported(m, levels, 4)) return 4;
  return 2;
}

// Copies, per problem, the order row of the current epoch into the buffer its
// captured minibatch kernels read.  One block per problem.
__global__ void __launch_bounds__(256) k_batch_orders(const int32_t* const* src, int32_t* const* dst, const int* n,
                                                      const int* epoch) {
  const int q = blockIdx.x;
  const int len = n[q];
  const int32_t* from = src[q] + (size_t)(*epoch) * len;
  for (int i = threadIdx.x; i < len; i += 256) dst[q][i] = from[i];
}

__global__ void k_epoch_advance(int* epoch) { *epoch += 1; }

cudaError_t launch_batch_orders(const int32_t* const* src, int32_t* const* dst, const int* n, int count,
                                const int* epoch, cudaStream_t s) {
  k_batch_orders<<<count, 256, 0, s>>>(src, dst, n, epoch);
  return cudaGetLastError();
}

cudaError_t launch_epoch_advance(int* epoch, cudaStream_t s) {
  k_epoch_advance<<<1, 1, 0, s>>>(epoch);
  return cudaGetLastError();
}

cudaError_t launch_apply(const ApplyArgs& a, cudaStream_t s) {
  const int n_tiles = a.tiles_x * a.tiles_y;
  const int n_probe = (a.m * a.m + kApplyProbePx - 1) / kApplyProbePx;
  const size_t bytes = (size_t)a.b * 3 * sizeof(int);
  cudaError_t e = launch_pdl(k_apply, dim3(n_tiles + n_probe), dim3(kApplyThreads), bytes, s, a);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

cudaError_t launch_misfit(int m, const float2* object, const float2* probe, const int32_t* pos,
                          const float* amp, int n_rows, int n_cols, int n_pos, double* partial,
                          cudaStream_t s) {
  FwdArgs f{};
  f.object = object;
  f.probe = probe;
  f.pos = pos;
  f.amp = amp;
  f.n_rows = n_rows;
  f.n_cols = n_cols;
  f.partial = partial;
  EMG_DISPATCH_M(m, (launch_forward_t<M, 0>(n_pos, f, s)));
}

cudaError_t launch_sum(const double* x, int n, double scale, double* out, cudaStream_t s) {
  k_sum<<<1, kSumThreads, 0, s>>>(x, n, scale, out);
  return cudaGetLastError();
}

cudaError_t launch_simulate(int m, const float2* object, const float2* probe, const int32_t* pos,
                            int n_rows, int n_cols, int n_pos, float* out, cudaStream_t s) {
  FwdArgs f{};
  f.object = object;
  f.probe = probe;
  f.pos = pos;
  f.n_rows = n_rows;
  f.n_cols = n_cols;
  f.out_intensity = out;
  EMG_DISPATCH_M(m, (launch_forward_t<M, 1>(n_pos, f, s)));
}

cudaError_t launch_fft2(int m, const float2* in, float2* out, int count, int inverse,
                        cudaStream_t s) {
  FwdArgs f{};
  f.in = in;
  f.out = out;
  if (inverse) EMG_DISPATCH_M(m, (launch_forward_t<M, 3>(count, f, s)));
  EMG_DISPATCH_M(m, (launch_forward_t<M, 2>(count, f, s)));
}

template <int M>
int gradient_wave_t() {
  using TL = WaveTile<M>;
  constexpr size_t bytes = gradc_smem_elems<M>() * sizeof(float2);
  int n = 0;
  cudaError_t e;
  if constexpr (TL::CTAS == 1) {
    int dev = 0, sms = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_gradc<M>, TL::NT, bytes);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    n *= sms;
  } else {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(TL::CTAS * 4096);
    cfg.blockDim = dim3(TL::NT);
    cfg.dynamicSmemBytes = bytes;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = TL::CTAS;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    e = cudaOccupancyMaxActiveClusters(&n, k_gradc<M>, &cfg);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

int gradient_slots(int m, int wave, int chunk) { return m <= 128 && wave > 0 && wave < chunk ? wave : chunk; }

int gradient_positions_per_wave(int m) {
  switch (m) {
    case 16: return gradient_wave_t<16>();
    case 32: return gradient_wave_t<32>();
    case 64: return gradient_wave_t<64>();
    case 128: return gradient_wave_t<128>();
    case 256: return gradient_wave_t<256>();
    default: return 0;
  }
}

cudaError_t launch_gradient(int m, int slots, int wave, const GradArgs& a, cudaStream_t s) {
  // m = 128 with at most half a wave of positions: clusters of 2, so that they spread over the SMs (us per
  // call without the misfit, one CTA against 2: 1 position 26.6 / 20.5, 38 30.8 / 22.6, 76 32.8 / 24.7)
  switch (m) {
    case 16: return launch_gradc_t<16>(slots, a, s);
    case 32: return launch_gradc_t<32>(slots, a, s);
    case 64: return launch_gradc_t<64>(slots, a, s);
    case 128: return 2 * slots <= wave ? launch_gradc_t<128, 2>(slots, a, s) : launch_gradc_t<128>(slots, a, s);
    case 256: return launch_gradc_t<256>(slots, a, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_grad_reduce(const GradReduceArgs& a, cudaStream_t s) {
  GradReduceArgs t = a;
  t.tiles_x = (a.n_cols + kGradTileW - 1) / kGradTileW;
  t.tiles_y = (a.n_rows + 2 * kGradTileH - 1) / (2 * kGradTileH);
  const int n_probe = (a.m * a.m + kApplyProbePx - 1) / kApplyProbePx;
  const bool small = t.tiles_x * t.tiles_y < kGradSmallTiles;
  if (small) t.tiles_y = (a.n_rows + kGradTileH - 1) / kGradTileH;
  const dim3 grid(t.tiles_x * t.tiles_y + n_probe);
  const cudaError_t e = small ? launch_pdl(k_grad_reduce<1, 8>, grid, dim3(kApplyThreads), 0, s, t)
                              : launch_pdl(k_grad_reduce<2, 4>, grid, dim3(kApplyThreads), 0, s, t);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// Whether the step kernel for probe side m with `cluster` CTAs per position
// supports `levels` multigrid levels.
bool step_supported(int m, int levels, int cluster) {
  const bool built = (cluster == 1 && m <= 32) || (cluster == 2 && m <= 128) || (cluster == 4 && (m == 64 || m == 128)) ||
                     (cluster == 8 && m >= 128);
  if (!built) return false;
  if ((m >> (levels - 1)) < cluster) return false;  // every CTA needs a row at the coarsest level
  size_t need = 0;
  for (int l = 1; l < levels; ++l) {
    const size_t wl = (size_t)m >> l, hl = wl / cluster;
    need += (2 * hl + 2) * (wl + 1);
  }
  // the buffers reuse the column slab (m = 256: an area sized for every level count that passes the row rule)
  return m == 256 || need <= (size_t)(m / cluster) * (m + 1);
}

cudaError_t launch_normalize_probe(const float* amp, int m, int n_pos, float2* probe,
                                   double* scratch, int scratch_len, cudaStream_t s) {
  const size_t n = (size_t)n_pos * m * m;
  int blocks = (int)((n + kNormThreads - 1) / kNormThreads);
  if (blocks > scratch_len) blocks = scratch_len;
  k_sum_sq<<<blocks, kNormThreads, 0, s>>>(amp, n, scratch);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_scale_probe<<<1, kScaleThreads, 0, s>>>(scratch, blocks, m, n_pos, probe);
  return cudaGetLastError();
}

}  // namespace emg

// ===========================================================================
// Allocation-free minibatch step: emg_step_minibatch_noalloc (include/emagpie.h).
//
// For callers that may not allocate device memory: code that runs inside a
// memory pool or arena it does not own, code that must not grow the device
// footprint after start-up, or code under a host-side policy that forbids
// cudaMalloc on its hot path.  They pass every input and output; the only
// scratch is the fixed array below, which every GPU that loads this library
// holds until the process exits.
// ===========================================================================
#include <string.h>

#include <mutex>

#include "../../include/emagpie.h"

namespace emg {
namespace {

static __device__ __align__(256) unsigned char g_noalloc_scratch[EMG_NOALLOC_SCRATCH_BYTES];

std::mutex g_noalloc_mu;
unsigned char* g_noalloc_base[256] = {nullptr};

struct NoAllocLayout {
  size_t idx, mq, wq, zt, qt, mu, phi, phi_after, total;
  size_t G[kMaxLevels], Q[kMaxLevels], u[kMaxLevels], Wz[kMaxLevels], WR[kMaxLevels], T[kMaxLevels];
};

// Byte offsets of every scratch array of one call, each 256-byte aligned.
NoAllocLayout noalloc_layout(int m, int levels, int b) {
  NoAllocLayout L{};
  size_t bytes = 0;
  auto take = [&](size_t n) {
    const size_t off = (bytes + 255) & ~(size_t)255;
    bytes = off + n;
    return off;
  };
  L.idx = take((size_t)b * sizeof(int32_t));
  L.mq = take(2 * sizeof(unsigned));
  for (int l = 0; l < levels; ++l) {
    const size_t n = (size_t)(m >> l) * (m >> l);
    L.G[l] = take(n * sizeof(float2));
    L.Q[l] = take(n * sizeof(float2));
    L.u[l] = take(n * sizeof(float));
    if (l + 1 < levels) {
      L.Wz[l] = take(n * sizeof(float));
      L.WR[l] = take(n * sizeof(float2));
      L.T[l] = take(n / 4 * sizeof(float));
    }
  }
  L.wq = take((size_t)m * m * sizeof(float));
  L.zt = take((size_t)b * m * m * sizeof(float2));
  L.qt = take((size_t)b * m * m * sizeof(float2));
  L.mu = take((size_t)b * sizeof(float));
  L.phi = take((size_t)b * sizeof(double));
  L.phi_after = take((size_t)b * sizeof(double));
  L.total = bytes;
  return L;
}

// Once per device, with that device current: twiddles, kernel attributes and
// the device address of the scratch array (a host-side name of a __device__
// array is not a device address, so it is looked up here).
cudaError_t noalloc_setup(int dev, unsigned char** base) {
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (dev < 0 || dev >= 256) return cudaErrorInvalidDevice;
  if (g_noalloc_base[dev]) {
    *base = g_noalloc_base[dev];
    return cudaSuccess;
  }
  cudaError_t e = upload_twiddles();
  if (e != cudaSuccess) return e;
  const int lim = step_smem_limit();
  if ((e = cudaFuncSetAttribute(k_step<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim)) ||
      (e = cudaFuncSetAttribute(k_step<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim)) ||
      (e = cudaFuncSetAttribute(k_step<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim)) ||
      (e = cudaFuncSetAttribute(k_step<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim)))
    return e;
  void* p = nullptr;
  e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
  if (e != cudaSuccess) return e;
  g_noalloc_base[dev] = (unsigned char*)p;
  *base = (unsigned char*)p;
  return cudaSuccess;
}

// The minibatch's position indices travel inside the seed kernel's launch parameters.
constexpr int kNoAllocMaxIdx = kSeedMaxIdx;

template <int M>
cudaError_t launch_step_natural(int b, const StepArgs& a, cudaStream_t s) {
  const size_t bytes = step_smem_elems<M>(a.levels) * sizeof(float2);
  k_step<M><<<b, StepThreads<M>::value, bytes, s>>>(a);
  return cudaGetLastError();
}

}  // namespace
}  // namespace emg

extern "C" emg_status emg_step_minibatch_noalloc(float* object, int32_t n_rows, int32_t n_cols,
                                                 float* probe, int32_t m, const int32_t* pos,
                                                 const float* intensity, int32_t n_pos,
                                                 const int32_t* idx, int32_t b,
                                                 const emg_params* p, emg_stream_t stream) {
  using namespace emg;
  if (!object || !probe || !pos || !intensity || !idx || !p) return EMG_EINVAL;
  if (n_rows < 1 || n_cols < 1 || n_pos < 1 || b < 1 || b > n_pos || b > kNoAllocMaxIdx) return EMG_EINVAL;
  if (m != 16 && m != 32 && m != 64 && m != 128) return EMG_ENOTSUP;  // m = 256 needs a cluster
  if (!(p->alpha > 0.f) || !isfinite(p->alpha) || !(p->w_eps >= 0.f) || !isfinite(p->w_eps))
    return EMG_EINVAL;
  if (p->levels < 1 || p->levels > kMaxLevels || (m >> (p->levels - 1)) < 2) return EMG_EINVAL;
  if (p->prolong != EMG_PROLONG_CONST && p->prolong != EMG_PROLONG_BILINEAR) return EMG_EINVAL;
  if (p->combine != EMG_COMBINE_WAVG && p->combine != EMG_COMBINE_SUM) return EMG_EINVAL;
  if (p->joint != 0 && p->joint != 1) return EMG_EINVAL;
  if (p->scatter != EMG_SCATTER_DETERMINISTIC) return EMG_ENOTSUP;
  if (p->dft != EMG_DFT_FFT32) return p->dft == EMG_DFT_BF16X3 ? EMG_ENOTSUP : EMG_EINVAL;
  if (step_smem_bytes(m, p->levels) > (size_t)step_smem_limit()) return EMG_ENOTSUP;
  for (int i = 0; i < b; ++i)
    if (idx[i] < 0 || idx[i] >= n_pos) return EMG_EINVAL;
  const NoAllocLayout L = noalloc_layout(m, p->levels, b);
  if (L.total > (size_t)EMG_NOALLOC_SCRATCH_BYTES) return EMG_EINVAL;  // beyond the fixed scratch

  int dev = 0;
  unsigned char* base = nullptr;
  if (cudaGetDevice(&dev) != cudaSuccess || noalloc_setup(dev, &base) != cudaSuccess) return EMG_ECUDA;
  const cudaStream_t s = (cudaStream_t)stream;
  int32_t* d_idx = (int32_t*)(base + L.idx);
  unsigned* d_mq = (unsigned*)(base + L.mq);
  if (launch_seed((const float2*)probe, m, d_mq, nullptr, d_idx, idx, b, s) != cudaSuccess) return EMG_ECUDA;

  PrepArgs pa{};
  StepArgs sa{};
  pa.probe = (const float2*)probe;
  pa.mq_read = d_mq;
  pa.mq_next = d_mq + 1;
  pa.m = m;
  pa.levels = p->levels;
  pa.prolong = p->prolong;
  pa.alpha = p->alpha;
  pa.w_eps = p->w_eps;
  pa.wq = (float*)(base + L.wq);
  for (int l = 0; l < p->levels; ++l) {
    pa.G[l] = (float2*)(base + L.G[l]);
    pa.Q[l] = (float2*)(base + L.Q[l]);
    pa.u[l] = (float*)(base + L.u[l]);
    sa.lv.G[l] = pa.G[l];
    sa.lv.Q[l] = pa.Q[l];
    if (l + 1 < p->levels) {
      pa.Wz[l] = (float*)(base + L.Wz[l]);
      pa.WR[l] = (float2*)(base + L.WR[l]);
      pa.T[l] = (float*)(base + L.T[l]);
      sa.lv.Wz[l] = pa.Wz[l];
      sa.lv.WR[l] = pa.WR[l];
    }
  }
  sa.object = (const float2*)object;
  sa.probe = (const float2*)probe;
  sa.pos = pos;
  sa.amp = intensity;
  sa.order = d_idx;
  sa.n_rows = n_rows;
  sa.n_cols = n_cols;
  sa.n_pos = n_pos;
  sa.b = b;
  sa.levels = p->levels;
  sa.prolong = p->prolong;
  sa.joint = p->joint;
  sa.verify = 0;
  sa.mq = d_mq;
  sa.zt = (float2*)(base + L.zt);
  sa.qt = (float2*)(base + L.qt);
  sa.mu = (float*)(base + L.mu);
  sa.phi = (double*)(base + L.phi);
  sa.phi_after = (double*)(base + L.phi_after);
  ApplyArgs aa{};
  aa.object = (float2*)object;
  aa.probe = (float2*)probe;
  aa.pos = pos;
  aa.order = d_idx;
  aa.b = b;
  aa.n_pos = n_pos;
  aa.n_rows = n_rows;
  aa.n_cols = n_cols;
  aa.m = m;
  aa.combine = p->combine;
  aa.zt = sa.zt;
  aa.qt = sa.qt;
  aa.mu = sa.mu;
  aa.wq = pa.wq;
  aa.mq_next = d_mq + 1;
  aa.tiles_x = apply_tiles_x(n_cols);
  aa.tiles_y = apply_tiles_y(n_rows);

  cudaError_t e = launch_prep(pa, false, s);
  if (e == cudaSuccess) {
    switch (m) {
      case 16: e = launch_step_natural<16>(b, sa, s); break;
      case 32: e = launch_step_natural<32>(b, sa, s); break;
      case 64: e = launch_step_natural<64>(b, sa, s); break;
      default: e = launch_step_natural<128>(b, sa, s); break;
    }
  }
  if (e == cudaSuccess) e = launch_apply(aa, s);
  return e == cudaSuccess ? EMG_OK : EMG_ECUDA;
}
