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
// of all ns, several shots' loads in flight; the copies move a piece of a row per warp
// with eight loads in flight per lane.  What bounds them is HBM and L2 (the record is
// read back from L2), and where few samples are blended the walk's latency.  256 shots x
// 64 receivers x 1024 samples, us: every sample checking every shot 1000, the list
// 29 (3.4 TB/s of shots and record, cold); one thread per sample 47 and 46, a row
// per warp 17 (pseudo-deblend) and 17 (sort, 7.9 TB/s of its bytes, partly L2).
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"

namespace ashrt {
namespace {

constexpr int kBThreads = 256;
constexpr int kBMaxShots = 8192;

constexpr int kBWarps = kBThreads / 32;

// grid (tiles over t', groups of receivers).  TX threads (32 to 256, a power of two)
// share a receiver and take NS samples each, TX apart; a CTA has 256 / TX receivers at a
// time and `per` times as many in all.  Shared: the shots whose window meets the tile,
// index and firing sample, in shot order (at most ns).
template <int NS>
__global__ void __launch_bounds__(kBThreads) k_blend(const float* __restrict__ D, int ns, int nr,
                                                     int nt, const int* __restrict__ fire,
                                                     float* __restrict__ b, int nb, int tx_n, int per) {
  const int TX = NS == 1 ? tx_n : kBThreads;     // (four samples: 256, immediate offsets)
  extern __shared__ int2 list[];
  __shared__ int counts[kBWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, tx = tid & (TX - 1);
  const long long tp0 = (long long)blockIdx.x * (TX * NS);
  int n = 0;
  for (int base = 0; base < ns; base += kBThreads) {
    const int i = base + tid;
    // some t' of the tile has 0 <= t' - fire[i] < nt
    const int fi = i < ns ? __ldg(fire + i) : 0;
    const bool in = i < ns && (long long)fi < tp0 + TX * NS && (long long)fi + nt > tp0;
    const unsigned m = __ballot_sync(0xffffffffu, in);
    if (lane == 0) counts[warp] = __popc(m);
    __syncthreads();
    int at = n;
#pragma unroll
    for (int w = 0; w < kBWarps; ++w) {
      if (w < warp) at += counts[w];
      n += counts[w];
    }
    if (in) list[at + __popc(m & ((1u << lane) - 1u))] = make_int2(i, fi);
    __syncthreads();
  }
  const int step = kBThreads / TX;
  const long long shot = (long long)nr * nt;
  const unsigned tp = (unsigned)tp0 + tx;
  int r = blockIdx.y * per * step + tid / TX;
  for (int k = 0; k < per && r < nr; ++k, r += step) {
    const float* rows = D + (long long)r * nt;
    float acc[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) acc[s] = 0.f;
    // the thread's sample of a listed shot, 0 where it has none (a listed shot is less than
    // nt and a tile away: 32 bits hold t' - fire, and a negative one is past nt)
    auto sample = [&](int2 e) {
      const unsigned t = tp - (unsigned)e.y;
      return t < (unsigned)nt ? __ldg(rows + e.x * shot + t) : 0.f;
    };
    if (NS == 1) {                                 // eight shots' loads in flight, then two
      int q = 0;
      for (; q + 8 <= n; q += 8) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = sample(list[q + u]);
#pragma unroll
        for (int u = 0; u < 8; ++u) acc[0] += v[u];
      }
      for (; q < n; q += 2) {
        const float v0 = sample(list[q]), v1 = q + 1 < n ? sample(list[q + 1]) : 0.f;
        acc[0] += v0;
        acc[0] += v1;
      }
    } else {                                       // (eight CTAs per SM hide the chain)
      for (int q = 0; q < n; ++q) {
        const int2 e = list[q];
        const float* row = rows + e.x * shot;
        const long long t0 = tp0 + tx - e.y;
#pragma unroll
        for (int s = 0; s < NS; ++s) {
          const long long t = t0 + s * TX;
          if (t >= 0 && t < nt) acc[s] += __ldg(row + t);
        }
      }
    }
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const long long at = tp0 + tx + s * TX;
      if (at < nb) b[(long long)r * nb + at] = acc[s];
    }
  }
}

// Rows that a copy's warps take in pieces of `len` elements, `segs` to a row.
struct Pieces {
  long long len;
  int segs;
};

// One warp per piece of a row of the shots [ns][nr][nt], eight samples per lane in flight.
// (WHOLE: one piece per row)
template <bool WHOLE>
__global__ void __launch_bounds__(kBThreads) k_pseudo_deblend(const float* __restrict__ b, int nr,
                                                              int nb, const int* __restrict__ fire,
                                                              int ns, int nt, Pieces pc,
                                                              float* __restrict__ D) {
  const int lane = threadIdx.x & 31;
  const long long all = (long long)ns * nr * (WHOLE ? 1 : pc.segs), stride = (long long)gridDim.x * kBWarps;
  for (long long p = (long long)blockIdx.x * kBWarps + (threadIdx.x >> 5); p < all; p += stride) {
    const long long q = WHOLE ? p : p / pc.segs, first = WHOLE ? 0 : (p - q * pc.segs) * pc.len;
    const long long end = WHOLE ? nt : min((long long)nt, first + pc.len);
    const int i = (int)(q / nr), r = (int)(q % nr);
    const long long f = __ldg(fire + i);
    const float* rec = b + (long long)r * nb;
    float* row = D + q * nt;
    for (long long t0 = first + lane; t0 < end; t0 += 256) {
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const long long t = t0 + 32 * k, tp = f + t;
        v[k] = (t < end && tp >= 0 && tp < nb) ? __ldg(rec + tp) : 0.f;
      }
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (t0 + 32 * k < end) row[t0 + 32 * k] = v[k];
    }
  }
}

// dst[j][i][:] = src[i][j][:], one warp per piece of a row of dst; V: float4 where every
// row starts on a 16-byte boundary, else float.  n: row length in V.
template <typename V, bool WHOLE>
__global__ void __launch_bounds__(kBThreads) k_sort(const V* __restrict__ src, int n0, int n1,
                                                    long long n, Pieces pc, V* __restrict__ dst) {
  const int lane = threadIdx.x & 31;
  const long long all = (long long)n0 * n1 * (WHOLE ? 1 : pc.segs), stride = (long long)gridDim.x * kBWarps;
  for (long long p = (long long)blockIdx.x * kBWarps + (threadIdx.x >> 5); p < all; p += stride) {
    const long long q = WHOLE ? p : p / pc.segs, first = WHOLE ? 0 : (p - q * pc.segs) * pc.len;
    const long long end = WHOLE ? n : min(n, first + pc.len);
    const long long j = q / n0, i = q % n0;
    const V* s = src + (i * n1 + j) * n;
    V* d = dst + q * n;
    for (long long t0 = first + lane; t0 < end; t0 += 256) {
      V v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (t0 + 32 * k < end) v[k] = __ldg(s + t0 + 32 * k);
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (t0 + 32 * k < end) d[t0 + 32 * k] = v[k];
    }
  }
}

// Rows of n elements are cut into pieces of whole 256s until there are 16 warps per SM:
// whole rows, where they are few and long, left the chip to a handful of warps (8 rows of
// a million samples, pseudo-deblend 1341 us whole and 10.3 in pieces, sort 644 and 8.2).
Pieces row_pieces(long long rows, long long n) {
  const long long chunks = (n + 255) / 256, warps = 152LL * 16;
  const long long want = std::min(chunks, (warps + rows - 1) / rows);
  Pieces p;
  p.len = (chunks + want - 1) / want * 256;
  p.segs = (int)((n + p.len - 1) / p.len);
  return p;
}

// CTAs of eight pieces, at most what keeps every SM full several times over
unsigned row_blocks(long long pieces) {
  const long long b = (pieces + kBWarps - 1) / kBWarps;
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
  // A record of at most 128 samples leaves threads for further receivers.  Four samples per
  // thread where two CTAs per SM remain, one otherwise (the walk over a long list is a
  // chain, so few samples want many threads: 64 shots x 64 receivers, all within 1024
  // samples, 18.4 us with four and 6.2 with one; 2048 shots x 1 within 512 461 and 83;
  // 512 shots x 8 receivers over 100000 samples, 784 CTAs, 18.5 and 26.8);
  // receivers share a CTA's list as long as eight waves remain.
  int TX = 256;
  while (TX > 32 && TX / 2 >= nb) TX /= 2;
  const long long groups = ((long long)nr * TX + kBThreads - 1) / kBThreads;
  auto tiles = [&](int NS) { return (long long)(nb - 1) / (TX * NS) + 1; };
  const bool four = TX == 256 && tiles(4) * groups >= 2LL * 152;
  const int per = tiles(four ? 4 : 1) * groups >= 8LL * 152 * 8 ? 4 : 1;
  const dim3 grid((unsigned)tiles(four ? 4 : 1), (unsigned)((groups + per - 1) / per));
  const size_t smem = ns * sizeof(int2);
  static SmemAttr attr1, attr4;
  const cudaError_t e = four ? set_smem(k_blend<4>, smem, attr4) : set_smem(k_blend<1>, smem, attr1);
  if (e != cudaSuccess) {
    set_error("ashrt_blend: %s", cudaGetErrorString(e));
    return ASHRT_ECUDA;
  }
  auto* kern = four ? k_blend<4> : k_blend<1>;
  kern<<<grid, kBThreads, smem, (cudaStream_t)stream>>>(shots_dev, ns, nr, nt, fire_dev, record_dev,
                                                        nb, TX, per);
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
  const long long rows = (long long)ns * nr;
  const Pieces pc = row_pieces(rows, nt);
  auto* kern = pc.segs == 1 ? k_pseudo_deblend<true> : k_pseudo_deblend<false>;
  kern<<<row_blocks(rows * pc.segs), kBThreads, 0, (cudaStream_t)stream>>>(
      record_dev, nr, nb, fire_dev, ns, nt, pc, shots_dev);
  return launched("ashrt_pseudo_deblend");
}

extern "C" ashrt_status ashrt_sort_gathers(const float* src_dev, int n0, int n1, int nt,
                                           float* dst_dev, void* stream) {
  if (!src_dev || !dst_dev || src_dev == dst_dev || n0 < 1 || n0 > 65535 || n1 < 1 ||
      n1 > 65535 || nt < 1) {
    set_error("ashrt_sort_gathers: need distinct arrays, 1 <= n0, n1 <= 65535, nt >= 1");
    return ASHRT_EINVAL;
  }
  const long long rows = (long long)n0 * n1;
  const bool vec = nt % 4 == 0 && (((uintptr_t)src_dev | (uintptr_t)dst_dev) & 15) == 0;
  const long long n = vec ? nt / 4 : nt;
  const Pieces pc = row_pieces(rows, n);
  const unsigned grid = row_blocks(rows * pc.segs);
  if (vec) {
    auto* kern = pc.segs == 1 ? k_sort<float4, true> : k_sort<float4, false>;
    kern<<<grid, kBThreads, 0, (cudaStream_t)stream>>>((const float4*)src_dev, n0, n1, n, pc,
                                                       (float4*)dst_dev);
  } else {
    auto* kern = pc.segs == 1 ? k_sort<float, true> : k_sort<float, false>;
    kern<<<grid, kBThreads, 0, (cudaStream_t)stream>>>(src_dev, n0, n1, n, pc, dst_dev);
  }
  return launched("ashrt_sort_gathers");
}
