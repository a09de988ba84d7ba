// Blending, pseudo-deblending and gather sorting (ch. 2, Eqs ch2_blending and
// pseudodeblending_equ): the acquisition model around the deblending solve.
//
//   blending        b[r, t'] = sum_i D[i, r, t' - tau_i]   (0 <= t' - tau_i < nt)
//   pseudo-deblend  D~[i, r, t] = b[r, tau_i + t]          (0 <= tau_i + t < nb, else 0)
//   sorting         [n0][n1][nt] -> [n1][n0][nt]           (shot <-> receiver gathers)
//
// D is the cube of common-shot gathers [ns][nr][nt], b one continuous record
// per receiver [nr][nb], tau_i the firing sample of shot i (whole samples; a
// device array).  Pseudo-deblending is the exact transpose of blending.
// Blending is written as a gather (each record sample sums the shots whose
// window covers it, in shot order), so it needs no atomics and its result
// does not depend on scheduling; the other two are copies.  All three are
// memory-bound streams with coalesced rows along t.
//
// A CTA of the blend lists the shots that reach its tile of the record once, in
// shot order, and its samples walk that list (about nt / spacing shots) instead
// of all ns; the copies move a row per warp with eight loads in flight per lane.
// What bounds them is HBM and L2 (the record is read back from L2).  256 shots x
// 64 receivers x 1024 samples, us: every sample checking every shot 1000, the list
// 29 (3.4 TB/s of shots and record, cold); one thread per sample 47 and 46, a row
// per warp 17 (pseudo-deblend) and 17 (sort, 7.9 TB/s of its bytes, partly L2).
#include <cuda_runtime.h>

#include "internal.h"

namespace ashrt {
namespace {

constexpr int kBThreads = 256;
constexpr int kBMaxShots = 8192;

constexpr int kBTile = 4 * kBThreads;   // record samples per CTA, four per thread

// grid (tiles over t', ceil(nr / per_cta)).  Shared: the indices of the shots
// whose window meets the tile, in shot order (at most ns).
__global__ void __launch_bounds__(kBThreads) k_blend(const float* __restrict__ D, int ns, int nr,
                                                     int nt, const int* __restrict__ fire,
                                                     float* __restrict__ b, int nb, int per_cta) {
  extern __shared__ int list[];
  __shared__ int counts[kBThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long tp0 = (long long)blockIdx.x * kBTile;
  int n = 0;
  for (int base = 0; base < ns; base += kBThreads) {
    const int i = base + tid;
    // some t' of the tile has 0 <= t' - fire[i] < nt
    const long long f = i < ns ? (long long)__ldg(fire + i) : 0;
    const bool in = i < ns && f < tp0 + kBTile && f + nt > tp0;
    const unsigned m = __ballot_sync(0xffffffffu, in);
    if (lane == 0) counts[warp] = __popc(m);
    __syncthreads();
    int at = n;
#pragma unroll
    for (int w = 0; w < kBThreads / 32; ++w) {
      if (w < warp) at += counts[w];
      n += counts[w];
    }
    if (in) list[at + __popc(m & ((1u << lane) - 1u))] = i;
    __syncthreads();
  }
  const int r1 = min(nr, ((int)blockIdx.y + 1) * per_cta);
  for (int r = blockIdx.y * per_cta; r < r1; ++r) {
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int q = 0; q < n; ++q) {
      const int i = list[q];
      const float* row = D + ((long long)i * nr + r) * nt;
      const long long t0 = tp0 + tid - __ldg(fire + i);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const long long t = t0 + k * kBThreads;
        if (t >= 0 && t < nt) acc[k] += __ldg(row + t);
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const long long tp = tp0 + tid + k * kBThreads;
      if (tp < nb) b[(long long)r * nb + tp] = acc[k];
    }
  }
}

// One warp per row of the shots [ns][nr][nt], eight samples per lane in flight.
__global__ void __launch_bounds__(kBThreads) k_pseudo_deblend(const float* __restrict__ b, int nr,
                                                              int nb, const int* __restrict__ fire,
                                                              int ns, int nt,
                                                              float* __restrict__ D) {
  const int lane = threadIdx.x & 31;
  const long long rows = (long long)ns * nr, stride = (long long)gridDim.x * (kBThreads / 32);
  for (long long q = (long long)blockIdx.x * (kBThreads / 32) + (threadIdx.x >> 5); q < rows;
       q += stride) {
    const int i = (int)(q / nr), r = (int)(q % nr);
    const long long f = __ldg(fire + i);
    const float* rec = b + (long long)r * nb;
    float* row = D + q * nt;
    for (long long t0 = lane; t0 < nt; t0 += 256) {
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const long long t = t0 + 32 * k, tp = f + t;
        v[k] = (t < nt && tp >= 0 && tp < nb) ? __ldg(rec + tp) : 0.f;
      }
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (t0 + 32 * k < nt) row[t0 + 32 * k] = v[k];
    }
  }
}

// dst[j][i][:] = src[i][j][:], one warp per row of dst; V: float4 where every row
// starts on a 16-byte boundary, else float.  n: row length in V.
template <typename V>
__global__ void __launch_bounds__(kBThreads) k_sort(const V* __restrict__ src, int n0, int n1,
                                                    long long n, V* __restrict__ dst) {
  const int lane = threadIdx.x & 31;
  const long long rows = (long long)n0 * n1, stride = (long long)gridDim.x * (kBThreads / 32);
  for (long long q = (long long)blockIdx.x * (kBThreads / 32) + (threadIdx.x >> 5); q < rows;
       q += stride) {
    const long long j = q / n0, i = q % n0;
    const V* s = src + (i * n1 + j) * n;
    V* d = dst + q * n;
    for (long long t0 = lane; t0 < n; t0 += 256) {
      V v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (t0 + 32 * k < n) v[k] = __ldg(s + t0 + 32 * k);
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (t0 + 32 * k < n) d[t0 + 32 * k] = v[k];
    }
  }
}

// CTAs of eight rows, at most what keeps every SM full several times over
unsigned row_blocks(long long rows) {
  const long long b = (rows + kBThreads / 32 - 1) / (kBThreads / 32);
  return (unsigned)(b > 152 * 64 ? 152 * 64 : b);
}

ashrt_status launched(const char* name) {
  count_launches(1);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error("%s: launch failed: %s", name, cudaGetErrorString(e));
    return ASHRT_ECUDA;
  }
  return ASHRT_OK;
}

}  // namespace
}  // namespace ashrt

using namespace ashrt;

extern "C" ashrt_status ashrt_blend(const float* shots_dev, int ns, int nr, int nt,
                                    const int* fire_dev, float* record_dev, int nb, void* stream) {
  if (!shots_dev || !fire_dev || !record_dev || ns < 1 || ns > kBMaxShots || nr < 1 ||
      nr > 65535 || nt < 1 || nb < 1) {
    set_error("ashrt_blend: need arrays, 1 <= ns <= %d, 1 <= nr <= 65535, nt >= 1, nb >= 1",
              kBMaxShots);
    return ASHRT_EINVAL;
  }
  // receivers per CTA share the list, as long as two waves of CTAs remain
  const unsigned tiles = (unsigned)((nb - 1) / kBTile + 1);
  const int per = (long long)tiles * nr >= 8LL * 152 * 8 ? 4 : 1;
  k_blend<<<dim3(tiles, (nr + per - 1) / per), kBThreads, ns * sizeof(int),
            (cudaStream_t)stream>>>(shots_dev, ns, nr, nt, fire_dev, record_dev, nb, per);
  return launched("ashrt_blend");
}

extern "C" ashrt_status ashrt_pseudo_deblend(const float* record_dev, int nr, int nb,
                                             const int* fire_dev, int ns, int nt,
                                             float* shots_dev, void* stream) {
  if (!record_dev || !fire_dev || !shots_dev || ns < 1 || ns > 65535 || nr < 1 || nr > 65535 ||
      nt < 1 || nb < 1) {
    set_error("ashrt_pseudo_deblend: need arrays, 1 <= ns, nr <= 65535, nt >= 1, nb >= 1");
    return ASHRT_EINVAL;
  }
  k_pseudo_deblend<<<row_blocks((long long)ns * nr), kBThreads, 0, (cudaStream_t)stream>>>(
      record_dev, nr, nb, fire_dev, ns, nt, shots_dev);
  return launched("ashrt_pseudo_deblend");
}

extern "C" ashrt_status ashrt_sort_gathers(const float* src_dev, int n0, int n1, int nt,
                                           float* dst_dev, void* stream) {
  if (!src_dev || !dst_dev || src_dev == dst_dev || n0 < 1 || n0 > 65535 || n1 < 1 ||
      n1 > 65535 || nt < 1) {
    set_error("ashrt_sort_gathers: need distinct arrays, 1 <= n0, n1 <= 65535, nt >= 1");
    return ASHRT_EINVAL;
  }
  const unsigned grid = row_blocks((long long)n0 * n1);
  if (nt % 4 == 0 && (((uintptr_t)src_dev | (uintptr_t)dst_dev) & 15) == 0)
    k_sort<float4><<<grid, kBThreads, 0, (cudaStream_t)stream>>>(
        (const float4*)src_dev, n0, n1, nt / 4, (float4*)dst_dev);
  else
    k_sort<float><<<grid, kBThreads, 0, (cudaStream_t)stream>>>(src_dev, n0, n1, nt, dst_dev);
  return launched("ashrt_sort_gathers");
}
