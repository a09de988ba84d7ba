// Trace-axis analysis (r2c) of panels whose traces fill at most half of the
// padded axis (nx <= N/2, the default padding): the transform of xfft.cu with
// the zero half taken out of the algorithm.
//
// With x[n] = 0 for n >= M = N/2, the spectrum splits into two length-M
// transforms of the same input,
//   X[2k]     = sum_{n < M} x[n] W_M^{nk},
//   X[2k + 1] = sum_{n < M} (x[n] W_N^n) W_M^{nk},       W_q = exp(-2 pi i / q).
// The factor W_N^n of the odd rows needs no pass of its own: in a pass of radix
// R over sub-transforms of length Ns the even rows' input r takes the twiddle
// W_{Ns R}^{k r}, the odd rows' W_{2 Ns R}^{(2k + 1) r} (in the first pass, Ns = 1,
// the constant W_{2R}^r; what is left of W_N^n is a common factor of a
// butterfly's inputs, which the next pass's twiddles take on).  Every thread
// holds 16 rows of a column, so M = 128 and 256 take two passes (16 x 8, 16 x 16)
// and M = 512 three (8 x 8 x 8), where the length-N transforms take three and
// four; the first pass reads no zeros, and the last one is in place without a
// barrier (its butterflies read and write the same elements).
//
// A CTA transforms 2 C adjacent time columns of one panel, packed two by two
// into complex columns (see xfft.cu), with M / 16 threads per packed column.
// The kernel streams its operands once (a third of the bytes read, two thirds
// written), so what counts is how many loads and stores an SM keeps in flight:
// the register cap below lets three 64 KB CTAs share an SM at N = 512 and 1024
// (with two, N = 1024: 291 us instead of 247).  Measured, us per launch, the
// length-N kernel and this one: 64 gathers x 32 panels of 256 x 1024 1490 / 1182
// (5.5 TB/s), 64 x 16 of 128 x 1024 353 / 283, 5 x 24 of 417 x 1500 306 / 247.
// A synthesis of the same form (nx <= N/2 kept, e + conj(W_N)^n o) crosses
// shared memory twice instead of four times but needs 107 registers for its
// mirrored rows, and two CTAs of eight warps hide its loads worse than the
// length-N kernel's sixteen (1302 against 1205 us): it is not used.
#include <cuda_runtime.h>

#include "stolt_r16.cuh"
#include "xfft_common.cuh"

namespace ashrt {

namespace {

// cos, sin of 2 pi r / 32, r = 0..15
__device__ constexpr float kCos32[16] = {
    1.f, 0.98078528040323044f, 0.92387953251128676f, 0.83146961230254524f,
    0.70710678118654752f, 0.55557023301960222f, 0.38268343236508977f, 0.19509032201612827f,
    0.f, -0.19509032201612827f, -0.38268343236508977f, -0.55557023301960222f,
    -0.70710678118654752f, -0.83146961230254524f, -0.92387953251128676f, -0.98078528040323044f};
__device__ constexpr float kSin32[16] = {
    0.f, 0.19509032201612827f, 0.38268343236508977f, 0.55557023301960222f,
    0.70710678118654752f, 0.83146961230254524f, 0.92387953251128676f, 0.98078528040323044f,
    1.f, 0.98078528040323044f, 0.92387953251128676f, 0.83146961230254524f,
    0.70710678118654752f, 0.55557023301960222f, 0.38268343236508977f, 0.19509032201612827f};

// exp(-2 pi i q / N), q < 64 (N 1024: 512), from the last pass's base-twiddle table of length N
template <int LOGN>
__device__ __forceinline__ float2 unit(const float2* __restrict__ tw, int q) {
  return base_twiddle<-1>(tw, Sched<LOGN>::tw_off(Sched<LOGN>::NPASS - 1), q);
}

// Resident CTAs per SM the kernel is compiled for.
template <int LOGN, int C, bool CG>
constexpr int r2c_half_minb() {
  return (LOGN >= 9 && !CG ? 768 : 512) / ((1 << LOGN) * C / 32);
}

// CG: with the fused CGLS update (XfftArgs::cg_mode), where the TMA kernel of
// xfft.cu does not apply (nx > 256 or rows that are not 16-byte aligned).
template <int LOGN, int C, bool CG>
__global__ void __launch_bounds__((1 << LOGN) * C / 32, r2c_half_minb<LOGN, C, CG>())
xfft_r2c_half(XfftArgs a) {
  constexpr int N = 1 << LOGN, M = N / 2, J = M / 16;
  constexpr int R1 = LOGN == 10 ? 8 : 16, NB1 = 16 / R1;   // first radix
  constexpr int RL = LOGN == 9 ? 16 : 8, NBL = 16 / RL;    // last radix
  static_assert(R1 * RL * (LOGN == 10 ? 8 : 1) == M, "N 256, 512 or 1024");
  extern __shared__ float2 sm[];   // even rows [M][C], odd rows [M][C]
  const int tid = threadIdx.x, col = tid % C, j = tid / C;
  const TileAt at = tile_at(a.nt, 2 * C);
  const long long slab = at.slab;
  const int ta = at.t0 + 2 * col;   // this thread packs columns ta (real) and ta + 1 (imag)
  const bool vec = (a.nt & 1) == 0;
  const float* in = a.in_real + slab * a.slab_real;
  const float* ew = a.ew ? a.ew + slab * a.slab_real : nullptr;
  const float* tm = a.tmask ? a.tmask + (slab / a.slabs_per_gather) * a.nx : nullptr;

  // The update's rows are loaded four at a time, each group's loads behind the stores
  // of the one before: all of the tile's rows are sent on their way into L2 first (8
  // gathers 1500 x 455, 24 panels, 987 -> 813 us; the next wave's tile as well or
  // instead: slower, its lines meet the stores of this one).
  if constexpr (CG) {
    const bool up = a.cg_mode == 1;
    const float4 cf = a.cg_coef[slab / a.slabs_per_gather];
    const bool two = up && a.cg_p2_read && cf.w != 0.f;
    const bool urw = up && a.cg_u_rw && (cf.z != 0.f || two);
    const long long o0 = slab * a.slab_real + at.t0;
    for (int row = tid; row < a.nx; row += M * C / 16) {
      const long long o = o0 + (long long)row * a.nt;
      prefetch_l2(a.cg_io + o);
      prefetch_l2(a.cg_s + o);
      if (urw) prefetch_l2(a.cg_u + o);
      if (two) prefetch_l2((a.cg_pout ? a.cg_pout : a.cg_io) + o);
    }
  }

  // first pass: butterfly jb = j + J q takes rows jb + r M / R1
  {
    float2 x[16];
    if constexpr (CG) {
      const float4 cf = a.cg_coef[slab / a.slabs_per_gather];
#pragma unroll
      for (int q = 0; q < NB1; ++q)
#pragma unroll
        for (int r = 0; r < R1; r += 4)
          cg_update_4(a, slab * a.slab_real, j + J * q + r * (M / R1), M / R1, ta, vec, cf,
                      x + q * R1 + r);
    } else {
#pragma unroll
      for (int q = 0; q < NB1; ++q)
#pragma unroll
        for (int r = 0; r < R1; ++r) {
          const int row = j + J * q + r * (M / R1);
          x[q * R1 + r] = row < a.nx ? load_pair_real(in + (long long)row * a.nt, ta, a.nt, vec)
                                     : make_float2(0.f, 0.f);
        }
    }
    if (ew || tm) {
#pragma unroll
      for (int q = 0; q < NB1; ++q)
#pragma unroll
        for (int r = 0; r < R1; ++r) {
          const int row = j + J * q + r * (M / R1);
          if (row < a.nx) {
            float2 w = ew ? load_pair_real(ew + (long long)row * a.nt, ta, a.nt, vec)
                          : make_float2(1.f, 1.f);
            const float g = tm ? __ldg(tm + row) : 1.f;
            x[q * R1 + r].x = x[q * R1 + r].x * w.x * g;
            x[q * R1 + r].y = x[q * R1 + r].y * w.y * g;
          }
        }
    }
#pragma unroll
    for (int q = 0; q < NB1; ++q) {
      float2 v[R1];
#pragma unroll
      for (int r = 0; r < R1; ++r) v[r] = x[q * R1 + r];
      dft16_r<-1, R1>(v);
#pragma unroll
      for (int r = 0; r < R1; ++r) sm[((j + J * q) * R1 + r) * C + col] = v[r];
#pragma unroll
      for (int r = 0; r < R1; ++r)
        v[r] = r == 0 ? x[q * R1]
                      : crot<-1>(x[q * R1 + r], kCos32[r * (16 / R1)], kSin32[r * (16 / R1)]);
      dft16_r<-1, R1>(v);
#pragma unroll
      for (int r = 0; r < R1; ++r) sm[(M + (j + J * q) * R1 + r) * C + col] = v[r];
    }
  }
  __syncthreads();

  if constexpr (LOGN == 10) {   // middle pass: radix 8 over sub-transforms of length 8
    constexpr int R = 8, Ns = 8;
#pragma unroll
    for (int odd = 0; odd < 2; ++odd) {
      float2* s = sm + odd * M * C;
      float2 v[16];
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int r = 0; r < R; ++r) v[q * R + r] = s[(j + J * q + r * (M / R)) * C + col];
      __syncthreads();
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int jb = j + J * q, k = jb & (Ns - 1);
        // W_{2 Ns R} = W_128 = W_N^8
        twiddle16_r<R>(v + q * R, unit<LOGN>(a.tw, (2 * k + odd) * (N / (2 * Ns * R))));
        dft16_r<-1, R>(v + q * R);
#pragma unroll
        for (int r = 0; r < R; ++r) s[((jb - k) * R + k + r * Ns) * C + col] = v[q * R + r];
      }
    }
    __syncthreads();
  }

  // last pass, in place: butterfly jb < M / RL reads and writes elements
  // jb + r M / RL
#pragma unroll
  for (int odd = 0; odd < 2; ++odd) {
    float2* s = sm + odd * M * C;
#pragma unroll
    for (int q = 0; q < NBL; ++q) {
      const int jb = j + J * q;
      float2 v[RL];
#pragma unroll
      for (int r = 0; r < RL; ++r) v[r] = s[(jb + r * (M / RL)) * C + col];
      twiddle16_r<RL>(v, unit<LOGN>(a.tw, 2 * jb + odd));
      dft16_r<-1, RL>(v);
#pragma unroll
      for (int r = 0; r < RL; ++r) s[(jb + r * (M / RL)) * C + col] = v[r];
    }
  }
  __syncthreads();

  // separate the packed columns (see xfft_r2c_kernel): thread (j, col) takes
  // rows j, j + J, ..., all of j's parity
  if (ta >= a.nt) return;
  const bool odd = j & 1, pair = ta + 1 < a.nt;
  const float2* s = sm + (odd ? M * C : 0) + col;
  float2* o = a.out_cplx + slab * a.slab_cplx + (long long)j * a.ld + ta;
  int k = j >> 1;                      // row l = 2 k + odd
#pragma unroll
  for (int i = 0; i <= 16; ++i) {      // the 17th, l = M, is thread j = 0's alone
    if (i < 16 || j == 0) {
      const float2 zl = s[(k & (M - 1)) * C];
      const float2 zm = s[(odd ? M - 1 - k : ((M - k) & (M - 1))) * C];
      const float4 AB = make_float4(0.5f * (zl.x + zm.x), 0.5f * (zl.y - zm.y),
                                    0.5f * (zl.y + zm.y), -0.5f * (zl.x - zm.x));
      if (pair) *(float4*)o = AB;
      else *o = make_float2(AB.x, AB.y);
    }
    k += J / 2;
    o += (long long)J * a.ld;
  }
}

template <int LOGN, int C, bool CG>
cudaError_t r2c_half_k(const XfftArgs& a, cudaStream_t s) {
  constexpr int T = (1 << LOGN) * C / 32;
  const size_t smem = (size_t)(1 << LOGN) * C * sizeof(float2);
  static SmemAttr attr;
  cudaError_t e = set_smem(xfft_r2c_half<LOGN, C, CG>, smem, attr);
  if (e != cudaSuccess) return e;
  xfft_r2c_half<LOGN, C, CG><<<tile_grid(a.slabs, a.nt, 2 * C), T, smem, s>>>(a);
  return cudaGetLastError();
}

template <int LOGN, int C>
cudaError_t r2c_half_v(const XfftArgs& a, cudaStream_t s) {
  return a.cg_mode ? r2c_half_k<LOGN, C, true>(a, s) : r2c_half_k<LOGN, C, false>(a, s);
}

}  // namespace

// Without the update at every launch size: 2 tiles 9.9 us length-N and 8.6 so, 256 tiles 12.8
// and 11.2 (N 512), 8064 tiles 220 and 176 (N 1024), at most 1.02 times in 195 launches.
// With the fused CGLS update from six waves of CTAs on: it has half the length-N
// kernel's threads per column, so with few tiles its groups of loads are a longer
// chain.  Both, us per launch (length-N, this): N 512, 18 / 90 / 900 / 1800 tiles 14 / 12 /
// 39 / 83 against 22 / 16 / 48 / 87; N 1024, 60 / 1200 / 1800 / 3600 tiles 14 / 58 / 90 /
// 227 against 23 / 67 / 95 / 178.
bool xfft_half_applies(const XfftArgs& a) {
  if (2 * a.nx > a.Nx || a.Nx < 256 || a.Nx > 1024) return false;
  if (!a.cg_mode) return true;
  const int c = a.Nx < 1024 && a.cols == 16 ? 16 : 8, res = 512 / (a.Nx * c / 32);
  return tile_grid(a.slabs, a.nt, 2 * c) >= 6u * 152u * (unsigned)res;
}

cudaError_t launch_xfft_r2c_half(const XfftArgs& a, cudaStream_t s) {
  switch (a.Nx) {
    case 256: return a.cols == 16 ? r2c_half_v<8, 16>(a, s) : r2c_half_v<8, 8>(a, s);
    case 512: return a.cols == 16 ? r2c_half_v<9, 16>(a, s) : r2c_half_v<9, 8>(a, s);
    default: return r2c_half_v<10, 8>(a, s);
  }
}

}  // namespace ashrt
