// Fused time-axis FFT + Stolt map + velocity/asymptote sum (forward) or
// spray (adjoint), one CTA per (gather pair, k_x) row.
//
// Forward, ch. 5 Eq. ch5_forward_operator / ch. 6 Eq. ch6_forward_operator,
// for the row of wavenumber index l of gather b:
//   for every panel p = (tau0_j, v_i):  load the x-transformed model row
//     X_p(l, tau) (nt samples), zero-pad to Nt, FFT along tau -> M_p(w_tau),
//     map w <- w_tau by the dispersion relation w_tau = sgn(w) sqrt(w^2 - (v k_x)^2)
//     (ch. 5) with linear interpolation, and accumulate
//     D(w) += exp(-i w tau0_j) V_p(w)   (T and the sums S / A)
//   D *= W(w) (wavelet C, band limit, 1/(Nt Nx)); inverse FFT along t; keep nt.
// Adjoint (ch. 5 Eq. ch5_adj_operator / ch. 6 Eq. ch6_adj_operator): the
// exact transpose: FFT the data row once, weight by W, and for each panel
// scatter every mapped bin to its two interpolation taps (transposed linear
// weights, conjugate phase), inverse FFT, keep nt samples.
//
// One CTA handles one k_x row of a PAIR of gathers, the two rows interleaved
// element by element (16-byte shared accesses; twiddles and Stolt taps
// computed once for both).  The panel spectrum, the map and the accumulation
// never leave the SM: the accumulator D lives in registers (each thread owns
// bins k = tid + T s), the spectrum of the current panel in one shared row,
// and the next panel's rows are staged with cp.async while the current one
// is transformed.
//
// The Stolt taps come from a table built on the host in FP64 (one word per
// (v, l, |k|): floor(u) and the 20-bit fraction of u = sqrt(k^2 - a^2), or
// "unmapped" when k^2 <= a^2), staged into shared memory with the panel, so
// the GPU and the FP64 oracle agree on cone membership and on the taps to
// 5e-7 in the interpolation weight.
#pragma once
#include <cuda_runtime.h>

#include <cmath>

#include "common.cuh"
#include "internal.h"

namespace ashrt {

struct Tap {
  int i0, i1;
  float w0, w1;
  bool valid;
};

// Interpolation taps of output bin k (natural index in [0, N)) from the tap
// word of |k|.  For w > 0 the taps are floor(u), floor(u)+1; for w < 0 the
// mirrored -floor(|u|), -floor(|u|)-1, which is the same linear interpolation
// at u = -|u| (odd extension keeps real output).  A tap on the w-Nyquist bin
// carries weight 0.
template <int N>
__device__ __forceinline__ Tap tap_decode(int k, unsigned w) {
  Tap t;
  t.valid = (k != N / 2) && (w != kTapInvalid);
  const int k0 = (int)(w >> 20);
  const float f = (float)(w & 0xfffffu) * (1.0f / 1048576.0f);
  if (k < N / 2) {
    t.i0 = k0;
    t.i1 = k0 + 1;
  } else {
    t.i0 = (N - k0) & (N - 1);
    t.i1 = (N - k0 - 1) & (N - 1);
  }
  t.w0 = 1.f - f;
  t.w1 = (t.i1 == N / 2) ? 0.f : f;
  return t;
}

template <int N>
__device__ __forceinline__ int kabs_of(int k) {
  return k <= N / 2 ? k : N - k;
}

// tap_decode for a bin whose side of the spectrum the caller knows: pos means
// k < N/2; otherwise k >= N/2 (the w-Nyquist bin k = N/2 is unmapped).  The
// row kernels' bins k = tid + T s lie on the positive side exactly for the
// first half of the slots s, so after unrolling `pos` is a constant and the
// side selection and the table index fold away.
template <int N>
__device__ __forceinline__ Tap tap_decode_side(int k, unsigned w, bool pos) {
  Tap t;
  t.valid = (pos || k != N / 2) && (w != kTapInvalid);
  const int k0 = (int)(w >> 20);
  const float f = (float)(w & 0xfffffu) * (1.0f / 1048576.0f);
  if (pos) {
    t.i0 = k0;
    t.i1 = k0 + 1;
  } else {
    t.i0 = (N - k0) & (N - 1);
    t.i1 = (N - k0 - 1) & (N - 1);
  }
  t.w0 = 1.f - f;
  t.w1 = (t.i1 == N / 2) ? 0.f : f;
  return t;
}

// Stage the rows of gathers A and B (B may be absent) of one panel: ld
// complex values each (ld is a multiple of 4, rows are 32-byte aligned).
__device__ __forceinline__ void stage_rows(float2* stage, const float2* rowA, const float2* rowB,
                                           int ld, int tid, int T) {
  const int chunks = ld >> 1;   // 16-byte chunks of two complex values
  for (int c = tid; c < chunks; c += T) cp_async16(stage + 2 * c, rowA + 2 * c);
  if (rowB)
    for (int c = tid; c < chunks; c += T) cp_async16(stage + ld + 2 * c, rowB + 2 * c);
}

// Stage one tap row (taps_ld words, a multiple of 4; 16-byte aligned).
__device__ __forceinline__ void stage_taps(unsigned* dst, const unsigned* src, int taps_ld, int tid,
                                           int T) {
  for (int c = tid; c < (taps_ld >> 2); c += T) cp_async16(dst + 4 * c, src + 4 * c);
}

// Stage one adjoint source-table row (n entries, n even; 16-byte aligned).
__device__ __forceinline__ void stage_tab(uint2* dst, const uint2* src, int n, int tid, int T) {
  for (int c = tid; c < (n >> 1); c += T) cp_async16(dst + 2 * c, src + 2 * c);
}

// Swizzle of a shared float4 row: XOR the 16-byte bank group (low 3 bits)
// with bits SW..SW+2 of the index (SW = 3: swz4 of common.cuh); SW = 0: no
// swizzle (a row written in natural order by consecutive lanes).
template <int SW>
__device__ __forceinline__ int swz_g(int i) {
  if constexpr (SW == 0) return i;
  else return i ^ ((i >> SW) & 7);
}

// One output bin j of the transposed Stolt map, gather form: the secondary
// source kB - 1 (weight f(kB - 1)) and the primary source kB (weight
// 1 - f(kB)) of |j| from the staged source-table row (see build_adj_table),
// on j's side of the spectrum; the w-Nyquist bin takes nothing.  dsp holds
// the weighted data spectrum; with SHIFT each source is multiplied by the
// conjugate asymptote phase of its own bin.
// pos: j < N/2 when the caller knows the side (see tap_decode_side), else
// j >= N/2.
template <int N, int SW, bool SHIFT>
__device__ __forceinline__ float4 adj_gather_bin(const float4* dsp, const uint2* stab, int j,
                                                 const float2* __restrict__ phj, bool pos) {
  constexpr int H = N / 2;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  if (!pos && j == H) return acc;
  const uint2 e = stab[pos ? j : N - j];
  const int kB = (int)(e.x >> 20);
  if (e.y & (1u << 21)) {
    const int kn = pos ? kB - 1 : N - kB + 1;
    float4 d = dsp[swz_g<SW>(kn)];
    if (SHIFT) d = cmul(d, cconj(__ldg(phj + kn)));
    acc = cscale(d, (float)(e.y & 0xfffffu) * (1.0f / 1048576.0f));
  }
  if (e.y & (1u << 20)) {
    const int kn = pos ? kB : N - kB;
    float4 d = dsp[swz_g<SW>(kn)];
    if (SHIFT) d = cmul(d, cconj(__ldg(phj + kn)));
    acc = cfma(1.f - (float)(e.x & 0xfffffu) * (1.0f / 1048576.0f), d, acc);
  }
  return acc;
}

// Bin 0 also takes the primary tap of -kB (w = 0 lies on both sides).
template <int N, int SW, bool SHIFT>
__device__ __forceinline__ float4 adj_gather_bin0_mirror(const float4* dsp, const uint2* stab,
                                                         const float2* __restrict__ phj, float4 acc) {
  const uint2 e = stab[0];
  if (e.y & (1u << 20)) {
    const int kn = N - (int)(e.x >> 20);
    float4 d = dsp[swz_g<SW>(kn)];
    if (SHIFT) d = cmul(d, cconj(__ldg(phj + kn)));
    acc = cfma(1.f - (float)(e.x & 0xfffffu) * (1.0f / 1048576.0f), d, acc);
  }
  return acc;
}

template <int N>
__device__ __forceinline__ void load_pair(float4* v, const float2* __restrict__ rowA,
                                          const float2* __restrict__ rowB, int nt, int tid) {
  constexpr int T = N / 8;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int i = tid + r * T;
    const float2 za = i < nt ? __ldg(rowA + i) : make_float2(0.f, 0.f);
    const float2 zb = (rowB && i < nt) ? __ldg(rowB + i) : make_float2(0.f, 0.f);
    v[r] = pack2(za, zb);
  }
}

// Shared bytes of the adjoint's source-table row (atab_row_len entries)
inline constexpr size_t adj_tab_bytes(int N) { return (size_t)(((N / 2 + 1) + 1) & ~1) * 8; }

// Largest dynamic shared memory a launch of the LOGN kernels may request
// (ld <= Nt, taps row <= Nt/2 + 4 words, source-table row Nt/2 + 2
// entries): the attribute is set once to it.
template <int LOGN>
inline size_t smem_cap(bool fwd) {
  constexpr int N = 1 << LOGN;
  const size_t taps = (size_t)(N / 2 + 4) * sizeof(unsigned);
  return fwd ? (size_t)N * sizeof(float4) + (size_t)2 * N * sizeof(float2) + 2 * taps
             : (size_t)2 * N * sizeof(float4) + adj_tab_bytes(N);
}

inline int row_log2(int n) {
  int l = 0;
  while ((1 << l) < n) ++l;
  return l;
}

// The panels [p0, p1) of chunk z when P panels are split into n chunks.
__device__ __forceinline__ void panel_chunk(int P, int n, int z, int& p0, int& p1) {
  const int per = (P + n - 1) / n;
  p0 = min(P, z * per);
  p1 = min(P, p0 + per);
}

// Chunks a row's panels are split into, so that few rows (small batches,
// narrow gathers) still fill the chip: 1, 2, 4 or 8.  `ctas` rows of P panels
// each run as ctas x n CTAs, `res` of them resident per SM.  With k CTAs on its SM a
// panel takes about (a^4 + k^4)^(1/4) times a constant: the latency of its dependent
// passes until `a` CTAs fill the pipe that bounds the kernel (shared memory or issue),
// its share of that pipe beyond.  A CTA costs about one and a half panels more (setup,
// and the extra data-row transform of the adjoint), and the forward's sum over the
// chunks (`sum`) as much again, so the candidate with the smallest
//   waves(n) (P / n + 1.5 [+ 1.5]) (a^4 + k(n)^4)^(1/4)
// is taken, if it is 5% below the unsplit one; waves(n) is the whole number, or with
// `ragged` the mean of it and the fraction (CTAs short enough to even out the last wave:
// adjoint, 1 gather 1024 x 417, 72 panels 435 -> 380 us).  With the residencies and the values
// of `a` at the launches, fitted to 1600 rows launches of 65 to 3084 rows, 1 to 32 panels
// and Nt 64 to 4096, the choice is within 1% of the best on average and at most 1.12 times
// the unsplit launch (a line in k without the sum's cost, as it was: 1.6 times, 26.7 and
// 41.9 us for 12 gathers 100 x 256, 9 panels).  `sum` (the forward) also splits up
// to eight panels one to a CTA or not at all, so that the partial sums, added in rank
// order, are those of the unsplit loop to the last bit.  Forward / adjoint rows per launch,
// whole and split: 1 gather 256 x 64, 8 panels (65 rows) 16.3 / 18.2 -> 11.0 / 10.4 us;
// 2 gathers 181 x 455, 25 panels (513 rows of pairs) 51 / 54 -> 45 / 41 us; 1 gather
// 1024 x 256, 32 panels (257 rows, single-gather form) 75 / 82 -> 62 / 60 us;
// 2 gathers 1024 x 128, 192 panels (258 rows) 451 / 555 -> 349 / 347 us, as 129
// pairs 459 -> 224 us forward.
inline int rows_split(long long ctas, int P, int res, double a, bool sum, bool ragged = false) {
  constexpr int kSms = 152;
  int best = 1;
  double best_t = 0.0;
  const bool whole = sum && P <= 8;
  for (int n = 1; n <= 8 && n <= P; n = whole && n < P ? P : 2 * n) {
    const double per_sm = (double)((ctas * n + kSms - 1) / kSms);
    const double k = per_sm < res ? per_sm : res;
    const double part = (double)(ctas * n) / kSms / k, whole_waves = std::ceil(per_sm / k);
    const double waves = ragged ? 0.5 * (whole_waves + (part > 1.0 ? part : 1.0)) : whole_waves;
    const double ends = sum && n > 1 ? 3.0 : 1.5;
    const double t = waves * ((P + n - 1) / n + ends) * std::pow(a * a * a * a + k * k * k * k, 0.25);
    if (n == 1 || t < (ragged ? 0.96 : 0.95) * best_t) {
      best = n;
      best_t = t;
    }
  }
  return best;
}

// Barrier of the thread-block cluster (all threads of all its CTAs).
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
  return r;
}
// 16 or 8 bytes of the same shared variable in the CTA of rank `rank`.
__device__ __forceinline__ unsigned cluster_addr(const void* p, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n"
               : "=r"(r)
               : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_load(unsigned a, float4& v) {
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];\n"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void cluster_load(unsigned a, float2& v) {
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];\n"
               : "=f"(v.x), "=f"(v.y)
               : "r"(a)
               : "memory");
}

__device__ __forceinline__ void cluster_store(unsigned a, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"r"(a), "f"(v.x), "f"(v.y),
               "f"(v.z), "f"(v.w)
               : "memory");
}
__device__ __forceinline__ void cluster_store(unsigned a, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};\n" ::"r"(a), "f"(v.x), "f"(v.y)
               : "memory");
}

// The forward's sum over the panel chunks of a row: the chunks' CTAs are one
// cluster, each leaves its V bins per thread (k = tid + T s) in its own shared
// row, and every CTA adds its share of the bins over all of them, in rank order
// (the sum does not depend on the scheduling), into rank 0's row.  The n loads
// of a bin are in flight together: rank 0 adding row after row takes 2.7 us
// longer for eight chunks at Nt 512.  Returns false in the other ranks, which
// are then done.
template <int V, int T, typename E>
__device__ __forceinline__ bool cluster_sum_rows(E* buf, E* acc, int tid, int n) {
  const unsigned rank = cluster_rank();
  __syncthreads();
#pragma unroll
  for (int s = 0; s < V; ++s) buf[tid + T * s] = acc[s];
  cluster_barrier();
  for (int k = (int)rank * T + tid; k < V * T; k += n * T) {
    E v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if (r < n) cluster_load(cluster_addr(buf + k, r), v[r]);
    E sum = v[0];
#pragma unroll
    for (int r = 1; r < 8; ++r)
      if (r < n) sum = cadd(sum, v[r]);
    cluster_store(cluster_addr(buf + k, 0), sum);
  }
  cluster_barrier();   // (also: a CTA's shared memory lives until the others have read it)
  if (rank != 0) return false;
#pragma unroll
  for (int s = 0; s < V; ++s) acc[s] = buf[tid + T * s];
  __syncthreads();     // every read of the row before the transform writes it
  return true;
}

// Launch of a kernel whose grid's z dimension is one cluster of n CTAs.
template <typename K, typename A>
inline cudaError_t launch_cluster_z(K kern, dim3 grid, int threads, size_t smem, int n,
                                    cudaStream_t s, const A& a) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = n;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

}  // namespace ashrt
