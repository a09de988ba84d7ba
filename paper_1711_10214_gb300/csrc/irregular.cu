// Traces at irregular positions (ch. 6: for non-uniformly sampled x the F
// operator is replaced by a discrete Fourier transform evaluated at the
// trace positions; ch. 5, ch. 6 cost discussion).
//
// The model keeps its regular apex grid x_a = j dx (the Stolt map needs it),
// so only the data side of the operator pair changes: the trace-axis
// synthesis of the forward, which the regular plan does with a c2r FFT from
// the half spectrum Y[l][t] (l = 0 .. Nx/2), becomes
//   d[j][t] = sum_l c_l Re( E[j][l] Y[l][t] ),   E[j][l] = exp(+2 pi i l x_j / (Nx dx)),
// with c_0 = c_{Nx/2} = 1 and c_l = 2 otherwise (the half spectrum of a real
// field; the Nyquist row enters as cos(pi x_j / dx)), and the adjoint's
// trace-axis analysis becomes its transpose
//   Yhat[l][t] = sum_j conj(E[j][l]) d[j][t].
// At x_j = j dx both reduce to the regular transforms.  The tables are built
// on the host in FP64 (c_l folded into the synthesis table).
//
// Both are dense complex contractions per gather, M x N x K = nr x nt x Lh
// and Lh x nt x nr, done here as FP32 tiled kernels on the CUDA cores, bound by
// their FP32 multiply-adds: 128 samples by 64 traces (32 wavenumbers) per CTA of
// 128 threads, 64 accumulators per thread in an outer product (each value read
// from shared memory serves 8 or 16 multiply-adds; with 16 accumulators the shared
// memory pipe was the bound), a half or a quarter of that where so large a tile leaves
// SMs idle, K in double-buffered chunks of eight with one barrier each.  The IRLS weights and the trace mask are fused into the synthesis epilogue
// (with the per-gather squared norm of the output for the CG scalars) and into the
// analysis operand load.  A sum runs over K in ascending order as before.
// 16 gathers 1024 x 256, 257 wavenumbers: 212 -> 123 us (35 TFLOP/s) and 162 ->
// 131 us (the 257th wavenumber's tile row included).
#include <cuda_runtime.h>

#include <cmath>
#include <vector>

#include "internal.h"

namespace ashrt {
namespace {

constexpr int kThr = 128, kBK = 8;   // 16 threads along the samples x 8

// n bytes from src, the rest of the 16, 8 or 4 zero
__device__ __forceinline__ void cp_zfill16(void* dst, const void* src, int n) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(n)
               : "memory");
}
__device__ __forceinline__ void cp_zfill8(void* dst, const void* src, int n) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(n)
               : "memory");
}
__device__ __forceinline__ void cp_zfill4(void* dst, const void* src, int n) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(n)
               : "memory");
}

__device__ __forceinline__ double warp_sum_dbl(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// d[g][j][t] = (sum_l Re(Es[j][l] Y[g][l][t])) * ew[g][j][t] * tmask[g][j];
// dot[g] += sum d^2.  RM traces x RN samples per thread; grid (ceil(nt/(16 RN)),
// ceil(nr/(8 RM)), batch).  Rows of Y are 16-byte aligned (ld a multiple of 4).
template <int RM, int RN>
__global__ void __launch_bounds__(kThr, 4) k_irr_synth(const float2* __restrict__ Es,
                                                       const float2* __restrict__ Y,
                                                       float* __restrict__ d, int nr, int nt, int Lh,
                                                       int ld, long long y_batch,
                                                       const float* __restrict__ ew,
                                                       const float* __restrict__ tmask,
                                                       double* __restrict__ dot) {
  constexpr int BM = 8 * RM, BN = 16 * RN;
  __shared__ __align__(16) float2 As[2][kBK][BM + 2];      // [l][j]
  __shared__ __align__(16) float2 Bs[2][kBK][BN];          // [l][t]
  // thread: traces ty RM .. + RM - 1, samples 2 tx + 32 q + {0, 1}
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int t0 = blockIdx.x * BN, j0 = blockIdx.y * BM, g = blockIdx.z;
  const float2* Yg = Y + (long long)g * y_batch;
  auto load = [&](int k0, int buf) {
#pragma unroll
    for (int u = 0; u < BM / 16; ++u) {        // eight l of a trace in adjacent threads
      const int kk = tid & 7, jj = (tid >> 3) + 16 * u, l = k0 + kk, j = j0 + jj;
      const bool in = j < nr && l < Lh;
      cp_zfill8(&As[buf][kk][jj], in ? Es + (long long)j * Lh + l : Es, in ? 8 : 0);
    }
#pragma unroll
    for (int u = 0; u < BN / 32; ++u) {        // two samples at a time, BN / 2 threads a row
      const int kk = tid / (BN / 2) + u * (256 / BN), tt = 2 * (tid & (BN / 2 - 1));
      const int l = k0 + kk, t = t0 + tt;
      const int n = l < Lh && t < nt ? (t + 1 < nt ? 16 : 8) : 0;
      cp_zfill16(&Bs[buf][kk][tt], n ? Yg + (long long)l * ld + t : Yg, n);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  float acc[RM][RN];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int q = 0; q < RN; ++q) acc[i][q] = 0.f;
  load(0, 0);
  for (int k0 = 0, buf = 0; k0 < Lh; k0 += kBK, buf ^= 1) {
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();   // this chunk is there; the other buffer's reads are done
    if (k0 + kBK < Lh) load(k0 + kBK, buf ^ 1);
#pragma unroll
    for (int k = 0; k < kBK; ++k) {
      float4 a[RM / 2], b[RN / 2];
#pragma unroll
      for (int i = 0; i < RM / 2; ++i) a[i] = *(const float4*)&As[buf][k][ty * RM + 2 * i];
#pragma unroll
      for (int q = 0; q < RN / 2; ++q) b[q] = *(const float4*)&Bs[buf][k][2 * tx + 32 * q];
#pragma unroll
      for (int i = 0; i < RM / 2; ++i)
#pragma unroll
        for (int q = 0; q < RN / 2; ++q) {
          float* c0 = &acc[2 * i][2 * q];
          float* c1 = &acc[2 * i + 1][2 * q];
          c0[0] = fmaf(a[i].x, b[q].x, fmaf(-a[i].y, b[q].y, c0[0]));
          c0[1] = fmaf(a[i].x, b[q].z, fmaf(-a[i].y, b[q].w, c0[1]));
          c1[0] = fmaf(a[i].z, b[q].x, fmaf(-a[i].w, b[q].y, c1[0]));
          c1[1] = fmaf(a[i].z, b[q].z, fmaf(-a[i].w, b[q].w, c1[1]));
        }
    }
  }
  double part = 0.0;
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    const int j = j0 + ty * RM + i;
    if (j >= nr) continue;
    const float tm = tmask ? __ldg(tmask + (long long)g * nr + j) : 1.f;
    const long long row = ((long long)g * nr + j) * nt;
    float p = 0.f;
#pragma unroll
    for (int q = 0; q < RN; ++q) {
      const int t = t0 + 2 * tx + 32 * (q >> 1) + (q & 1);
      if (t >= nt) continue;
      float v = acc[i][q] * tm;
      if (ew) v *= __ldg(ew + row + t);
      d[row + t] = v;
      p = fmaf(v, v, p);
    }
    part += (double)p;
  }
  if (dot) {
    __shared__ double red[kThr / 32];
    double p = warp_sum_dbl(part);
    if ((tid & 31) == 0) red[tid >> 5] = p;
    __syncthreads();
    if (tid < 32) {
      p = tid < kThr / 32 ? red[tid] : 0.0;
      p = warp_sum_dbl(p);
      if (tid == 0 && p != 0.0) atomicAdd(dot + g, p);
    }
  }
}

// Yhat[g][l][t] = sum_j Ea[l][j] (d[g][j][t] * ew[g][j][t] * tmask[g][j]),
// Ea = conj(E)^T.  RM wavenumbers x RN samples per thread; grid (ceil(nt/(16 RN)),
// ceil(Lh/(8 RM)), batch).  There is always one wavenumber more than a multiple of 32
// (Nx >= 64): a warp without any skips the multiply-adds.
template <int RM, int RN>
__global__ void __launch_bounds__(kThr, 4) k_irr_analysis(const float2* __restrict__ Ea,
                                                          const float* __restrict__ d,
                                                          float2* __restrict__ Yh, int nr, int nt,
                                                          int Lh, int ld, long long y_batch,
                                                          const float* __restrict__ ew,
                                                          const float* __restrict__ tmask) {
  constexpr int BM = 8 * RM, BN = 16 * RN;
  __shared__ __align__(16) float2 As[2][kBK][BM + 2];      // [j][l]
  __shared__ __align__(16) float Bs[2][kBK][BN];           // [j][t]
  __shared__ float Ws[2][kBK][BN];                         // [j][t]: ew
  // thread: wavenumbers RM ty .. + RM - 1, samples 4 tx + 64 h + 0 .. 3
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int t0 = blockIdx.x * BN, l0 = blockIdx.y * BM, g = blockIdx.z;
  const bool work = l0 + 2 * RM * (tid >> 5) < Lh;
  // (copied past the registers: the compiler moves register loads down to their use)
  float tmn = 1.f;                             // the mask of the trace that the thread copies
  auto load = [&](int k0, int buf) {
#pragma unroll
    for (int u = 0; u < BM / 16; ++u) {
      const int e = tid * (BM / 16), ll = e >> 3, kk = (e & 7) + u, l = l0 + ll, j = k0 + kk;
      const bool in = l < Lh && j < nr;
      cp_zfill8(&As[buf][kk][ll], in ? Ea + (long long)l * nr + j : Ea, in ? 8 : 0);
    }
    const int j = k0 + ty;
    if (tmask) tmn = j < nr ? __ldg(tmask + (long long)g * nr + j) : 1.f;
    const long long row = ((long long)g * nr + j) * nt;
#pragma unroll
    for (int u = 0; u < RN; ++u) {
      const int t = t0 + tx + 16 * u;
      const bool in = j < nr && t < nt;
      cp_zfill4(&Bs[buf][ty][tx + 16 * u], in ? d + row + t : d, in ? 4 : 0);
      if (ew) cp_zfill4(&Ws[buf][ty][tx + 16 * u], in ? ew + row + t : ew, in ? 4 : 0);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  float2 acc[RM][RN];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int q = 0; q < RN; ++q) acc[i][q] = make_float2(0.f, 0.f);
  load(0, 0);
  for (int k0 = 0, buf = 0; k0 < nr; k0 += kBK, buf ^= 1) {
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    if (tmask || ew) {                         // the thread's own copies
#pragma unroll
      for (int u = 0; u < RN; ++u) {
        float& v = Bs[buf][ty][tx + 16 * u];
        v *= tmn;
        if (ew) v *= Ws[buf][ty][tx + 16 * u];
      }
    }
    __syncthreads();   // this chunk is there; the other buffer's reads are done
    if (k0 + kBK < nr) load(k0 + kBK, buf ^ 1);
    if (work) {
#pragma unroll
      for (int k = 0; k < kBK; ++k) {
        float4 a[RM / 2], b[RN / 4];
#pragma unroll
        for (int i = 0; i < RM / 2; ++i) a[i] = *(const float4*)&As[buf][k][ty * RM + 2 * i];
#pragma unroll
        for (int h = 0; h < RN / 4; ++h) b[h] = *(const float4*)&Bs[buf][k][4 * tx + 64 * h];
#pragma unroll
        for (int i = 0; i < RM / 2; ++i)
#pragma unroll
          for (int q = 0; q < RN; ++q) {
            const float4 bv = b[q >> 2];
            const float v = (q & 3) == 0 ? bv.x : (q & 3) == 1 ? bv.y : (q & 3) == 2 ? bv.z : bv.w;
            acc[2 * i][q].x = fmaf(a[i].x, v, acc[2 * i][q].x);
            acc[2 * i][q].y = fmaf(a[i].y, v, acc[2 * i][q].y);
            acc[2 * i + 1][q].x = fmaf(a[i].z, v, acc[2 * i + 1][q].x);
            acc[2 * i + 1][q].y = fmaf(a[i].w, v, acc[2 * i + 1][q].y);
          }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    const int l = l0 + ty * RM + i;
    if (l >= Lh) continue;
    float2* out = Yh + (long long)g * y_batch + (long long)l * ld;
#pragma unroll
    for (int q = 0; q < RN; ++q) {
      const int t = t0 + 4 * tx + 64 * (q >> 2) + (q & 3);
      if (t < nt) out[t] = acc[i][q];
    }
  }
}

// r -= alpha q on the data side (the CGLS update the regular adjoint fuses
// into its trace-axis transform), per gather alpha = coef[g].z.
__global__ void k_irr_cg_r(float* __restrict__ r, const float* __restrict__ q, long long n,
                           const float4* __restrict__ coef) {
  const int g = blockIdx.y;
  const float a = coef[g].z;
  const long long off = (long long)g * n;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    r[off + i] = fmaf(-a, q[off + i], r[off + i]);
}

}  // namespace

bool build_irregular_tables(const double* x, int nr, int Nx, double dx, float2* Es, float2* Ea) {
  const int Lh = Nx / 2 + 1;
  for (int j = 0; j < nr; ++j) {
    if (!std::isfinite(x[j])) return false;
    for (int l = 0; l < Lh; ++l) {
      double re, im;
      if (l == Nx / 2) {
        re = std::cos(M_PI * x[j] / dx);
        im = 0.0;
      } else {
        // reduce the phase l x / (Nx dx) modulo 1 before scaling by 2 pi
        double ph = (double)l * x[j] / ((double)Nx * dx);
        ph -= std::floor(ph);
        re = std::cos(2.0 * M_PI * ph);
        im = std::sin(2.0 * M_PI * ph);
      }
      const double c = (l == 0 || l == Nx / 2) ? 1.0 : 2.0;
      Es[(size_t)j * Lh + l] = make_float2((float)(c * re), (float)(c * im));
      Ea[(size_t)l * nr + j] = make_float2((float)re, (float)(-im));
    }
  }
  return true;
}

// The tile of a launch over `rows` x nt outputs per gather: the fewest rounds of CTAs per
// SM times what one takes against the largest tile's (half the tile does a little more than
// half the time, as each value read from shared memory serves fewer multiply-adds).
struct IrrTile {
  int m, n;
  double cost;
};
static int irr_tile(const IrrTile (&tiles)[3], int rows, int nt, int batch) {
  int best = 0;
  double best_t = 0.0;
  for (int i = 0; i < 3; ++i) {
    const long long ctas = (long long)((nt + tiles[i].n - 1) / tiles[i].n) *
                           ((rows + tiles[i].m - 1) / tiles[i].m) * batch;
    const double t = (double)((ctas + 151) / 152) * tiles[i].cost;
    if (i == 0 || t < 0.95 * best_t) {
      best = i;
      best_t = t;
    }
  }
  return best;
}

// (us, the largest tile and the choice: 1 gather, 250 apexes, 300 traces x 1000 samples
// synthesis 42.6 and 26.6, analysis 30.9 and 20.7; 3 gathers, 30 apexes, 20 traces x 130
// samples synthesis 14.6 and 8.0; 16 gathers, 400 apexes, 63 traces x 130 samples analysis
// 27.2 and 22.7.)
cudaError_t launch_irr_synth(const float2* Es, const float2* Y, float* d, int nr, int nt, int Lh,
                             int ld, long long y_batch, const float* ew, const float* tmask,
                             double* dot, int batch, cudaStream_t s) {
  static constexpr IrrTile tiles[3] = {{64, 128, 1.0}, {64, 64, 0.6}, {32, 64, 0.4}};
  const int i = irr_tile(tiles, nr, nt, batch);
  const dim3 grid((nt + tiles[i].n - 1) / tiles[i].n, (nr + tiles[i].m - 1) / tiles[i].m, batch);
  auto* kern = i == 0 ? k_irr_synth<8, 8> : i == 1 ? k_irr_synth<8, 4> : k_irr_synth<4, 4>;
  kern<<<grid, kThr, 0, s>>>(Es, Y, d, nr, nt, Lh, ld, y_batch, ew, tmask, dot);
  return cudaGetLastError();
}

cudaError_t launch_irr_analysis(const float2* Ea, const float* d, float2* Yh, int nr, int nt,
                                int Lh, int ld, long long y_batch, const float* ew,
                                const float* tmask, int batch, cudaStream_t s) {
  static constexpr IrrTile tiles[3] = {{32, 128, 1.0}, {32, 64, 0.6}, {16, 64, 0.4}};
  const int i = irr_tile(tiles, Lh, nt, batch);
  const dim3 grid((nt + tiles[i].n - 1) / tiles[i].n, (Lh + tiles[i].m - 1) / tiles[i].m, batch);
  auto* kern = i == 0 ? k_irr_analysis<4, 8> : i == 1 ? k_irr_analysis<4, 4> : k_irr_analysis<2, 4>;
  kern<<<grid, kThr, 0, s>>>(Ea, d, Yh, nr, nt, Lh, ld, y_batch, ew, tmask);
  return cudaGetLastError();
}

cudaError_t launch_irr_cg_r(float* r, const float* q, long long n, const float4* coef, int batch,
                            cudaStream_t s) {
  long long gx = (n + 256 * 8 - 1) / (256 * 8);
  if (gx > 1024) gx = 1024;
  k_irr_cg_r<<<dim3((unsigned)(gx < 1 ? 1 : gx), batch), 256, 0, s>>>(r, q, n, coef);
  return cudaGetLastError();
}

}  // namespace ashrt
