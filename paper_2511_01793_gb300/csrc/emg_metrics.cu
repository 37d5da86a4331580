// FP64 reductions of the reconstruction quality on the GPU.
//
// Blind ptychography recovers (z, Q) only up to the scaling (c z, Q / c),
// c complex and non-zero: the exit waves Q . P_k z, and with them the data of
// Sec. 2.1, do not change.  A reconstruction is therefore compared with a
// reference after the best c over a region of the object (the pixels the
// scan illuminates well):
//
//   c = <z, z_ref> / <z, z>        (sums over the region; <a, b> = sum conj(a) b)
//   object error = ||c z - z_ref|| / ||z_ref||            (over the region)
//   probe error  = ||Q / c - Q_ref|| / ||Q_ref||          (whole probe)
//   phase RMS    = sqrt(mean over the region of arg(c z conj(z_ref))^2)
//
// and the region is { p : sum_k |Q_ref(p - o_k)|^2 >= frac * max }, the summed
// illumination of the scan (the paper's figures compare reconstructions over
// the scanned field, Sec. 4.1).
//
// Every sum is taken in FP64.  Each kernel uses a fixed grid and a fixed
// reduction tree, and the partial sums are added in a fixed order, so results
// are bitwise repeatable.  The illumination of a pixel is summed over the
// positions in index order, as a sequential loop would.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <mutex>

#include "../../include/emagpie.h"
#include "emg_internal.h"

namespace emg {
namespace {

constexpr int kMetThreads = 256;
constexpr int kMetBlocks = 304;  // 2 per SM on 152 SMs; fixed, so the sums are repeatable
constexpr int kPosChunk = 512;   // positions staged in shared memory at a time

// Scratch of one call, from a stream-ordered pool of this library (one per
// device): cudaMalloc and cudaFree cost more than the reductions themselves
// (512^2 pixels, m = 128, us per call with them / from the pool: region 173 / 79,
// errors 205 / 89).  The driver orders reuse between streams and threads; the pool
// keeps at most kScratchKeep bytes between calls and gives them back when a
// context on the device is destroyed.
constexpr size_t kScratchKeep = (size_t)64 << 20;
std::mutex g_scratch_mu;
cudaMemPool_t g_scratch_pool[256] = {nullptr};

cudaError_t scratch_alloc(double** p, size_t words, cudaStream_t s) {
  *p = nullptr;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess && (dev < 0 || dev >= 256)) e = cudaErrorInvalidDevice;
  cudaMemPool_t pool = nullptr;
  if (e == cudaSuccess) {
    std::lock_guard<std::mutex> lk(g_scratch_mu);
    if (!g_scratch_pool[dev]) {
      cudaMemPoolProps props = {};
      props.allocType = cudaMemAllocationTypePinned;
      props.location.type = cudaMemLocationTypeDevice;
      props.location.id = dev;
      cudaMemPool_t made = nullptr;
      unsigned long long keep = kScratchKeep;
      e = cudaMemPoolCreate(&made, &props);
      if (e == cudaSuccess) {
        e = cudaMemPoolSetAttribute(made, cudaMemPoolAttrReleaseThreshold, &keep);
        if (e == cudaSuccess)
          g_scratch_pool[dev] = made;
        else
          cudaMemPoolDestroy(made);
      }
    }
    pool = g_scratch_pool[dev];
  }
  if (e == cudaSuccess) e = cudaMallocFromPoolAsync((void**)p, words * sizeof(double), pool, s);
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}

// The block's sums of N quantities into out[0..N): shuffle trees, then the
// warps' values in warp order (one barrier for all of them).
template <int N>
__device__ __forceinline__ void block_sums(const double (&v)[N], double* out) {
  __shared__ double sh[N][kMetThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int j = 0; j < N; ++j) {
    double s = v[j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) sh[j][warp] = s;
  }
  __syncthreads();
  if (threadIdx.x < N) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kMetThreads / 32; ++w) s += sh[threadIdx.x][w];
    out[threadIdx.x] = s;
  }
}

// Partial sums over the region: |z|^2, conj(z) z_ref (re, im), |z_ref|^2, count.
__global__ void __launch_bounds__(kMetThreads) k_align_pass1(const float2* __restrict__ z,
                                                             const float2* __restrict__ zr,
                                                             const uint8_t* __restrict__ region, size_t n,
                                                             double* __restrict__ part) {
  double zz = 0.0, cr = 0.0, ci = 0.0, rr = 0.0, cnt = 0.0;
  for (size_t i = (size_t)blockIdx.x * kMetThreads + threadIdx.x; i < n; i += (size_t)gridDim.x * kMetThreads) {
    if (region && !region[i]) continue;
    const float2 a = z[i], b = zr[i];
    const double ax = a.x, ay = a.y, bx = b.x, by = b.y;
    zz += ax * ax + ay * ay;
    cr += ax * bx + ay * by;  // conj(a) b
    ci += ax * by - ay * bx;
    rr += bx * bx + by * by;
    cnt += 1.0;
  }
  const double v[5] = {zz, cr, ci, rr, cnt};
  block_sums(v, part + (size_t)blockIdx.x * 5);
}

// Sum of the kMetBlocks partials of one quantity (stride `words`) by one warp:
// a fixed number per lane in block order, then a shuffle tree.  (One thread
// that walked all partials took 90 us: a chain of dependent FP64 adds on loads.)
__device__ __forceinline__ double warp_sum_partials(const double* part, int words) {
  double s = 0.0;
#pragma unroll
  for (int i = 0; i < (kMetBlocks + 31) / 32; ++i) {
    const int b = i * 32 + (threadIdx.x & 31);
    if (b < kMetBlocks) s += part[(size_t)b * words];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// c = <z, z_ref> / <z, z> into res[0..1]; res[2] = ||z_ref||^2, res[3] = count.
// One warp per summed quantity.
__global__ void __launch_bounds__(160) k_align_final1(const double* __restrict__ part, double* __restrict__ res) {
  __shared__ double s[5];
  const int w = threadIdx.x >> 5;
  const double v = warp_sum_partials(part + w, 5);
  if ((threadIdx.x & 31) == 0) s[w] = v;
  __syncthreads();
  if (threadIdx.x != 0) return;
  res[0] = s[0] > 0.0 ? s[1] / s[0] : 0.0;
  res[1] = s[0] > 0.0 ? s[2] / s[0] : 0.0;
  res[2] = s[3];
  res[3] = s[4];
}

// Partial sums: |c z - z_ref|^2 and arg(c z conj(z_ref))^2 over the region,
// and (blocks covering the probe) |Q / c - Q_ref|^2, |Q_ref|^2.
__global__ void __launch_bounds__(kMetThreads) k_align_pass2(const float2* __restrict__ z,
                                                             const float2* __restrict__ zr,
                                                             const uint8_t* __restrict__ region, size_t n,
                                                             const float2* __restrict__ q,
                                                             const float2* __restrict__ qr, size_t nq,
                                                             const double* __restrict__ res,
                                                             double* __restrict__ part) {
  const double c_x = res[0], c_y = res[1];
  double e_obj = 0.0, e_ph = 0.0, e_q = 0.0, q_rr = 0.0;
  const size_t stride = (size_t)gridDim.x * kMetThreads;
  for (size_t i = (size_t)blockIdx.x * kMetThreads + threadIdx.x; i < n; i += stride) {
    if (region && !region[i]) continue;
    const float2 a = z[i], b = zr[i];
    const double wx = c_x * a.x - c_y * a.y, wy = c_x * a.y + c_y * a.x;  // c z
    const double dx = wx - b.x, dy = wy - b.y;
    e_obj += dx * dx + dy * dy;
    const double px = wx * b.x + wy * b.y, py = wy * b.x - wx * b.y;   // c z conj(z_ref)
    const double ph = atan2(py, px);
    e_ph += ph * ph;
  }
  const double cc = c_x * c_x + c_y * c_y;
  for (size_t i = (size_t)blockIdx.x * kMetThreads + threadIdx.x; i < nq; i += stride) {
    const float2 a = q[i], b = qr[i];
    // Q / c = Q conj(c) / |c|^2
    const double wx = cc > 0.0 ? (a.x * c_x + a.y * c_y) / cc : 0.0;
    const double wy = cc > 0.0 ? (a.y * c_x - a.x * c_y) / cc : 0.0;
    const double dx = wx - b.x, dy = wy - b.y;
    e_q += dx * dx + dy * dy;
    q_rr += (double)b.x * b.x + (double)b.y * b.y;
  }
  const double v[4] = {e_obj, e_ph, e_q, q_rr};
  block_sums(v, part + (size_t)blockIdx.x * 4);
}

__global__ void __launch_bounds__(128) k_align_final2(const double* __restrict__ part, double* __restrict__ res) {
  __shared__ double s[4];
  const int w = threadIdx.x >> 5;
  const double v = warp_sum_partials(part + w, 4);
  if ((threadIdx.x & 31) == 0) s[w] = v;
  __syncthreads();
  if (threadIdx.x != 0) return;
  const double rr = res[2], cnt = res[3];
  res[4] = rr > 0.0 ? sqrt(s[0] / rr) : 0.0;
  res[5] = s[3] > 0.0 ? sqrt(s[2] / s[3]) : 0.0;
  res[6] = cnt > 0.0 ? sqrt(s[1] / cnt) : 0.0;
}

// |Q_ref|^2 in FP64 (both products are exact); also clears the maximum.
__global__ void __launch_bounds__(kMetThreads) k_probe_intensity(const float2* __restrict__ qr, size_t n,
                                                                 double* __restrict__ p2,
                                                                 unsigned long long* __restrict__ max_bits) {
  const size_t first = (size_t)blockIdx.x * kMetThreads + threadIdx.x;
  if (first == 0) *max_bits = 0ull;
  for (size_t i = first; i < n; i += (size_t)gridDim.x * kMetThreads)
    p2[i] = (double)qr[i].x * qr[i].x + (double)qr[i].y * qr[i].y;
}

// Summed illumination of each object pixel, positions in index order, and the
// largest value (as bits: no value is negative).  One block per tile of 8 x 32
// pixels: the positions whose patch overlaps the tile are first gathered, in
// order, into a list, so a pixel walks only those instead of every position;
// |Q|^2 comes from a table, which leaves one FP64 add per covered pixel and
// position (the FP64 pipe is the bound: 23 us for 14.7 M of them).  512^2 pixels,
// 900 positions, m = 128, whole call: 79 us, with every position tested at every
// pixel 2380.
constexpr int kIllumRows = 8, kIllumCols = 32, kIllumWarps = kMetThreads / 32;
__global__ void __launch_bounds__(kMetThreads) k_illumination(const double* __restrict__ p2, int m,
                                                              const int32_t* __restrict__ pos, int n_pos,
                                                              int n_rows, int n_cols, int tiles_x,
                                                              double* __restrict__ illum,
                                                              unsigned long long* __restrict__ max_bits) {
  __shared__ int2 list[kPosChunk];
  __shared__ int count[kIllumWarps];
  __shared__ double warp_max[kIllumWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r0 = (int)(blockIdx.x / tiles_x) * kIllumRows, c0 = (int)(blockIdx.x % tiles_x) * kIllumCols;
  const int r = r0 + warp, c = c0 + lane;
  const bool live = r < n_rows && c < n_cols;
  double s = 0.0;
  constexpr int PW = kPosChunk / kIllumWarps, ROUNDS = PW / 32;  // positions of a chunk per warp
  for (int k0 = 0; k0 < n_pos; k0 += kPosChunk) {
    // ordered compaction: warp w takes the w-th run of the chunk's positions
    int2 p[ROUNDS];
    unsigned mask[ROUNDS];
    int mine = 0;
#pragma unroll
    for (int i = 0; i < ROUNDS; ++i) {
      const int k = k0 + warp * PW + i * 32 + lane;
      bool hit = false;
      if (k < n_pos) {
        p[i] = make_int2(pos[2 * k], pos[2 * k + 1]);
        hit = p[i].x < (long long)r0 + kIllumRows && (long long)p[i].x + m > r0 &&
              p[i].y < (long long)c0 + kIllumCols && (long long)p[i].y + m > c0;
      }
      mask[i] = __ballot_sync(0xffffffffu, hit);
      mine += __popc(mask[i]);
    }
    __syncthreads();  // the previous chunk's list has been walked
    if (lane == 0) count[warp] = mine;
    __syncthreads();
    int at = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kIllumWarps; ++w) {
      if (w < warp) at += count[w];
      total += count[w];
    }
#pragma unroll
    for (int i = 0; i < ROUNDS; ++i) {
      if (mask[i] >> lane & 1u) list[at + __popc(mask[i] & ((1u << lane) - 1u))] = p[i];
      at += __popc(mask[i]);
    }
    __syncthreads();
    if (live) {
      // the loads of eight positions in flight, the sums in order; 0 where the patch does not reach
      for (int j0 = 0; j0 < total; j0 += 8) {
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          v[u] = 0.0;
          if (j0 + u < total) {
            const int lr = r - list[j0 + u].x, lc = c - list[j0 + u].y;
            if ((unsigned)lr < (unsigned)m && (unsigned)lc < (unsigned)m) v[u] = p2[(size_t)lr * m + lc];
          }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) s += v[u];
      }
    }
  }
  if (live) illum[(size_t)r * n_cols + c] = s;
  double mx = live ? fmax(s, 0.0) : 0.0;  // fmax: a NaN never becomes the maximum
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) warp_max[warp] = mx;
  __syncthreads();
  if (tid == 0) {
#pragma unroll
    for (int w = 0; w < kIllumWarps; ++w) mx = fmax(mx, warp_max[w]);
    atomicMax(max_bits, (unsigned long long)__double_as_longlong(mx));
  }
}

__global__ void __launch_bounds__(kMetThreads) k_region_mask(const double* __restrict__ illum, size_t n,
                                                             const unsigned long long* __restrict__ max_bits,
                                                             double frac, uint8_t* __restrict__ region) {
  const double thr = frac * __longlong_as_double((long long)*max_bits);
  for (size_t i = (size_t)blockIdx.x * kMetThreads + threadIdx.x; i < n; i += (size_t)gridDim.x * kMetThreads)
    region[i] = illum[i] >= thr ? 1 : 0;
}

}  // namespace

void scratch_trim(int dev) {
  std::lock_guard<std::mutex> lk(g_scratch_mu);
  if (dev >= 0 && dev < 256 && g_scratch_pool[dev]) cudaMemPoolTrimTo(g_scratch_pool[dev], 0);
}

}  // namespace emg

extern "C" emg_status emg_aligned_errors(const float* object, const float* object_ref, int32_t n_rows,
                                         int32_t n_cols, const float* probe, const float* probe_ref, int32_t m,
                                         const uint8_t* region, double* out, emg_stream_t stream) {
  using namespace emg;
  if (!object || !object_ref || !probe || !probe_ref || !out || n_rows < 1 || n_cols < 1 || m < 1)
    return EMG_EINVAL;
  const cudaStream_t s = (cudaStream_t)stream;
  const size_t n = (size_t)n_rows * n_cols, nq = (size_t)m * m;
  double* scratch = nullptr;  // 5 + 4 partials per block, then 7 results
  if (scratch_alloc(&scratch, (size_t)kMetBlocks * 9 + 8, s) != cudaSuccess) return EMG_ENOMEM;
  double* p1 = scratch;
  double* p2 = scratch + (size_t)kMetBlocks * 5;
  double* res = scratch + (size_t)kMetBlocks * 9;
  double host[7];
  cudaError_t e = cudaSuccess;
  k_align_pass1<<<kMetBlocks, kMetThreads, 0, s>>>((const float2*)object, (const float2*)object_ref, region, n, p1);
  if ((e = cudaGetLastError()) == cudaSuccess) {
    k_align_final1<<<1, 160, 0, s>>>(p1, res);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    k_align_pass2<<<kMetBlocks, kMetThreads, 0, s>>>((const float2*)object, (const float2*)object_ref, region, n,
                                                     (const float2*)probe, (const float2*)probe_ref, nq, res, p2);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    k_align_final2<<<1, 128, 0, s>>>(p2, res);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(host, res, sizeof(host), cudaMemcpyDeviceToHost, s);
  const cudaError_t ef = cudaFreeAsync(scratch, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess || ef != cudaSuccess) return EMG_ECUDA;
  out[0] = host[0];  // c (re, im)
  out[1] = host[1];
  out[2] = host[4];  // object relative error
  out[3] = host[5];  // probe relative error
  out[4] = host[6];  // RMS phase difference
  return EMG_OK;
}

extern "C" emg_status emg_illuminated_region(const float* probe_ref, int32_t m, const int32_t* pos, int32_t n_pos,
                                             int32_t n_rows, int32_t n_cols, double frac, uint8_t* region,
                                             emg_stream_t stream) {
  using namespace emg;
  if (!probe_ref || !pos || !region || m < 1 || n_pos < 1 || n_rows < 1 || n_cols < 1 || !(frac >= 0.0) ||
      !isfinite(frac))
    return EMG_EINVAL;
  const cudaStream_t s = (cudaStream_t)stream;
  const size_t n = (size_t)n_rows * n_cols, nq = (size_t)m * m;
  const size_t tiles_x = ((size_t)n_cols + kIllumCols - 1) / kIllumCols;
  const size_t tiles_y = ((size_t)n_rows + kIllumRows - 1) / kIllumRows;
  double* scratch = nullptr;  // illumination, |Q_ref|^2, the maximum
  if (scratch_alloc(&scratch, n + nq + 1, s) != cudaSuccess) return EMG_ENOMEM;
  double* p2 = scratch + n;
  unsigned long long* max_bits = (unsigned long long*)(p2 + nq);
  k_probe_intensity<<<kMetBlocks, kMetThreads, 0, s>>>((const float2*)probe_ref, nq, p2, max_bits);
  k_illumination<<<(unsigned)(tiles_x * tiles_y), kMetThreads, 0, s>>>(p2, m, pos, n_pos, n_rows, n_cols, (int)tiles_x,
                                                                      scratch, max_bits);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) {
    k_region_mask<<<kMetBlocks, kMetThreads, 0, s>>>(scratch, n, max_bits, frac, region);
    e = cudaGetLastError();
  }
  const cudaError_t ef = cudaFreeAsync(scratch, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  return e == cudaSuccess && ef == cudaSuccess ? EMG_OK : EMG_ECUDA;
}
