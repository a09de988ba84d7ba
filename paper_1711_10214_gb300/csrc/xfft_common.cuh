// Loads, stores and reductions shared by the trace-axis transforms (xfft.cu,
// xfft_half.cu).
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"
#include "internal.h"

namespace ashrt {

// The panel and the first of the `cols` time columns of a CTA.  Consecutive
// CTAs take adjacent tiles of one panel, not the same tile of consecutive
// panels: the CTAs in flight then read and write neighbouring segments (128
// and 256 bytes) of the same rows, which stay together in L2 and in DRAM pages.
struct TileAt {
  unsigned slab;
  int t0;
};
__device__ __forceinline__ TileAt tile_at(unsigned block, int nt, int cols) {
  const unsigned n = (unsigned)(nt + cols - 1) / (unsigned)cols;
  TileAt at;
  at.slab = block / n;
  at.t0 = (int)(block % n) * cols;
  return at;
}
__device__ __forceinline__ TileAt tile_at(int nt, int cols) { return tile_at(blockIdx.x, nt, cols); }

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p));
}
inline unsigned tile_grid(int slabs, int nt, int cols) {
  return (unsigned)slabs * (unsigned)((nt + cols - 1) / cols);
}

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// Adds the CTA-wide sum of `part` to *dst (one atomic per CTA).
__device__ __forceinline__ void block_accumulate(double part, double* dst) {
  __shared__ double red[32];
  part = warp_sum(part);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) red[w] = part;
  __syncthreads();
  if (w == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    double x = lane < nw ? red[lane] : 0.0;
    x = warp_sum(x);
    if (lane == 0) atomicAdd(dst, x);
  }
}

// Real time samples t and t+1 of one trace, packed as z = x_t + i x_{t+1}
// (one 8-byte load when the row is 8-byte aligned).
__device__ __forceinline__ float2 load_pair_real(const float* __restrict__ row, int t, int nt,
                                                 bool vec) {
  if (vec && t + 1 < nt) return __ldg((const float2*)(row + t));
  return make_float2(t < nt ? __ldg(row + t) : 0.f, t + 1 < nt ? __ldg(row + t + 1) : 0.f);
}

// Plain (coherent) pair load / store of samples t, t+1 of a row, for the
// in-place CGLS updates (each pair is read and written by one thread).
__device__ __forceinline__ float2 ld_pair(const float* row, int t, int nt, bool vec) {
  if (vec && t + 1 < nt) return *(const float2*)(row + t);
  return make_float2(t < nt ? row[t] : 0.f, t + 1 < nt ? row[t + 1] : 0.f);
}

__device__ __forceinline__ void st_pair(float* row, int t, int nt, bool vec, float2 v) {
  if (vec && t + 1 < nt) {
    *(float2*)(row + t) = v;
    return;
  }
  if (t < nt) row[t] = v.x;
  if (t + 1 < nt) row[t + 1] = v.y;
}

// The fused CGLS update of one sample pair (see XfftArgs::cg_mode); returns
// the updated vector's pair, which is what the transform consumes.
__device__ __forceinline__ float2 cg_update_pair(const XfftArgs& a, long long off, int t, bool vec,
                                                 float4 cf) {
  float* io = a.cg_io + off;
  const float2 x = ld_pair(io, t, a.nt, vec);
  const float2 y = ld_pair(a.cg_s + off, t, a.nt, vec);
  float2 z;
  if (a.cg_mode == 1) {
    float* po = a.cg_pout ? a.cg_pout + off : io;
    z = make_float2(fmaf(cf.x, y.x, cf.y * x.x), fmaf(cf.x, y.y, cf.y * x.y));
    const bool two = a.cg_p2_read && cf.w != 0.f;
    if (a.cg_u_rw && (cf.z != 0.f || two)) {
      float* u = a.cg_u + off;
      float2 un = ld_pair(u, t, a.nt, vec);
      if (two) {
        const float2 p2 = ld_pair(po, t, a.nt, vec);   // read before z overwrites it
        un = make_float2(fmaf(cf.w, p2.x, un.x), fmaf(cf.w, p2.y, un.y));
      }
      un = make_float2(fmaf(cf.z, x.x, un.x), fmaf(cf.z, x.y, un.y));
      st_pair(u, t, a.nt, vec, un);
    }
    st_pair(po, t, a.nt, vec, z);
  } else {
    z = make_float2(fmaf(-cf.z, y.x, x.x), fmaf(-cf.z, y.y, x.y));
    st_pair(io, t, a.nt, vec, z);
  }
  return z;
}

// The fused CGLS update of the sample pairs of rows row, row + step, ..,
// row + 3 step (zeros where a row is >= nx), with every load before the first
// store: in-place updates row by row would make each row's loads wait for the
// stores of the one before.
__device__ __forceinline__ void cg_update_4(const XfftArgs& a, long long off, int row, int step,
                                            int t, bool vec, float4 cf, float2* z) {
  const float2 zero = make_float2(0.f, 0.f);
  const bool up = a.cg_mode == 1;
  const bool two = up && a.cg_p2_read && cf.w != 0.f;
  const bool urw = up && a.cg_u_rw && (cf.z != 0.f || two);
  float* dst = up && a.cg_pout ? a.cg_pout : a.cg_io;
  float2 x[4], y[4], u[4], p2[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const bool ok = row + i * step < a.nx;
    const long long o = off + (long long)(row + i * step) * a.nt;
    x[i] = ok ? ld_pair(a.cg_io + o, t, a.nt, vec) : zero;
    y[i] = ok ? ld_pair(a.cg_s + o, t, a.nt, vec) : zero;
    u[i] = ok && urw ? ld_pair(a.cg_u + o, t, a.nt, vec) : zero;
    p2[i] = ok && two ? ld_pair(dst + o, t, a.nt, vec) : zero;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const bool ok = row + i * step < a.nx;
    const long long o = off + (long long)(row + i * step) * a.nt;
    if (up) {
      z[i] = make_float2(fmaf(cf.x, y[i].x, cf.y * x[i].x), fmaf(cf.x, y[i].y, cf.y * x[i].y));
      if (urw && ok) {
        float2 un = u[i];
        if (two) un = make_float2(fmaf(cf.w, p2[i].x, un.x), fmaf(cf.w, p2[i].y, un.y));
        un = make_float2(fmaf(cf.z, x[i].x, un.x), fmaf(cf.z, x[i].y, un.y));
        st_pair(a.cg_u + o, t, a.nt, vec, un);
      }
    } else {
      z[i] = make_float2(fmaf(-cf.z, y[i].x, x[i].x), fmaf(-cf.z, y[i].y, x[i].y));
    }
    if (ok) st_pair(dst + o, t, a.nt, vec, z[i]);
  }
}

// Stored row `row` (<= N/2) of the half spectrum for the two adjacent columns
// t and t+1 (t even): (A, B) = (re, im of column t, re, im of column t+1).
// Rows are ld >= nt long with ld a multiple of 4, so the 16-byte load at an
// even t < nt stays inside the row; a column >= nt reads as zero.
__device__ __forceinline__ float4 col_load2(const float2* __restrict__ base, int ld, int row, int t,
                                            int nt) {
  const bool ok = t < nt, okb = t + 1 < nt;
  const float4 y = __ldg((const float4*)(base + (long long)row * ld + (ok ? t : 0)));
  return make_float4(ok ? y.x : 0.f, ok ? y.y : 0.f, okb ? y.z : 0.f, okb ? y.w : 0.f);
}
// Z = A + i B of a stored row (zdir), of its mirror N - row, whose A and B
// are the conjugates (zmir), and of rows 0 and N/2, whose imaginary parts a
// real signal's spectrum does not have (zreal).
__device__ __forceinline__ float2 zdir(float4 y) { return make_float2(y.x - y.w, y.y + y.z); }
__device__ __forceinline__ float2 zmir(float4 y) { return make_float2(y.x + y.w, y.z - y.y); }
__device__ __forceinline__ float2 zreal(float4 y) { return make_float2(y.x, y.z); }

}  // namespace ashrt
