// Learned warm start: a 4-level U-Net (the same architecture as the FP64
// reference of the tests) with hand-written forward and backward kernels.
// BF16 storage for weights and activations, FP32 accumulation, FP32 master
// weights and gradients, Adam.  It maps a pseudo-deblended gather to an
// initial Radon model (P channels) and initial IRLS residual weights
// (log W_r, one channel) for the warm-started robust solve.
//
// Layouts: activations NHWC (image rows = traces x, columns = time t, so a
// gather [nx][nt] is an nx x nt image) with a per-tensor pixel stride and
// channel offset, so skip connections are written straight into the channel
// slice of the concatenation buffer they feed.  Convolution weights are kept
// in FP32 "OIHW" order (the reference's order) and converted every step to the
// BF16 copies that the layer's kernels read (WCopies).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "internal.h"

namespace {

using bf16 = __nv_bfloat16;

template <typename T>
__device__ __forceinline__ void st_f(T* p, long long i, float v);
template <>
__device__ __forceinline__ void st_f<float>(float* p, long long i, float v) { p[i] = v; }
template <>
__device__ __forceinline__ void st_f<bf16>(bf16* p, long long i, float v) { p[i] = __float2bfloat16(v); }

struct Tensor {        // a channel slice of an NHWC buffer
  void* p = nullptr;
  int ps = 0;          // channels allocated per pixel
  int off = 0;         // first channel of the slice
};

// 2x2 average pooling (forward, bf16; 8 channels per thread, as k_up).
__global__ void __launch_bounds__(256) k_pool(Tensor in, Tensor out, int N, int H, int W, int C) {
  const int Ho = H / 2, Wo = W / 2, C8 = C / 8;
  const long long total = (long long)N * Ho * Wo * C8;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % C8) * 8;
    const long long p = i / C8;
    const int xo = (int)(p % Wo);
    const long long q = (2 * (p / Wo)) * W + 2 * xo;       // p / Wo = n Ho + yo, H even
    const bf16* src = (const bf16*)in.p + in.off + c;
    __align__(16) bf16 v[4][8], o[8];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      *(uint4*)v[k] = *(const uint4*)(src + (q + (k >> 1) * W + (k & 1)) * in.ps);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float s = 0.f;
#pragma unroll
      for (int k = 0; k < 4; ++k) s += __bfloat162float(v[k][j]);
      o[j] = __float2bfloat16(0.25f * s);
    }
    *(uint4*)((bf16*)out.p + p * out.ps + out.off + c) = *(const uint4*)o;
  }
}

// nearest 2x upsampling (forward, bf16; 8 channels = 16 bytes per thread, C,
// strides and offsets multiples of 8)
__global__ void k_up(Tensor in, Tensor out, int N, int H, int W, int C) {   // H, W: output sizes
  const int C8 = C / 8;
  const long long total = (long long)N * H * W * C8;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % C8) * 8;
    const long long p = i / C8;
    const int x = (int)(p % W);
    const long long ny = p / W;                 // n * H + y
    const int y = (int)(ny % H);
    const long long n = ny / H;
    const long long q = (n * (H / 2) + y / 2) * (W / 2) + x / 2;
    *(uint4*)((bf16*)out.p + p * out.ps + out.off + c) =
        *(const uint4*)((const bf16*)in.p + q * in.ps + in.off + c);
  }
}

// gathers [N][nx][nt] -> bf16 image [N][nx][nt][1] scaled by 1/rms[n]
__global__ void k_pack_in(const float* d, const float* rms, bf16* x, long long per, int N) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < per * N;
       i += (long long)gridDim.x * blockDim.x)
    x[i] = __float2bfloat16(d[i] / rms[i / per]);
}

// sum of squares of every gather, many CTAs per gather (FP64 throughout: a gather's
// amplitudes may be anywhere in FP32's range, and their squares are not; one atomic
// per CTA), then rms = sqrt(sum / per)
__global__ void k_sumsq(const float* d, long long per, double* acc) {
  const int n = blockIdx.y;
  double s = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < per;
       i += (long long)gridDim.x * blockDim.x) {
    const double v = d[n * per + i];
    s = fma(v, v, s);
  }
  __shared__ double red[256];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicAdd(acc + n, red[0]);
}

__global__ void k_rms_fin(const double* acc, long long per, float* rms, int N) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n < N) rms[n] = (float)fmax(sqrt(acc[n] / (double)per), 1e-30);
}

// First layer (one input channel -> 16): a thread takes four pixels of a row (W is
// a multiple of 8), so that each weight read from shared memory serves four
// products; the 3 x 6 neighbourhood comes from the BF16 image, 16 BF16 outputs per
// pixel leave as two 16-byte vectors (out.ps, out.off multiples of 8).
__global__ void __launch_bounds__(256) k_conv_first(const bf16* x, const bf16* w, const float* bias,
                                                    Tensor out, int N, int H, int W, int relu) {
  __shared__ __align__(16) float ws[9][16];
  __shared__ float bs[16];
  if (threadIdx.x < 144) ws[threadIdx.x / 16][threadIdx.x % 16] = __bfloat162float(w[threadIdx.x]);
  if (threadIdx.x < 16) bs[threadIdx.x] = bias[threadIdx.x];
  __syncthreads();
  const int W4 = W / 4;
  const long long total = (long long)N * H * W4;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int x0 = (int)(i % W4) * 4;
    const long long ny = i / W4;
    const int y = (int)(ny % H);
    float v[3][6];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const bool ok = y + r >= 1 && y + r <= H;
      const bf16* row = x + (ny + (ok ? r - 1 : 0)) * W + x0;
      __align__(8) bf16 m[4];
      *(uint2*)m = *(const uint2*)row;
      v[r][0] = ok && x0 > 0 ? __bfloat162float(row[-1]) : 0.f;
      v[r][5] = ok && x0 + 4 < W ? __bfloat162float(row[4]) : 0.f;
#pragma unroll
      for (int k = 0; k < 4; ++k) v[r][1 + k] = ok ? __bfloat162float(m[k]) : 0.f;
    }
    float acc[4][16];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int c = 0; c < 16; ++c) acc[k][c] = bs[c];
#pragma unroll
    for (int t = 0; t < 9; ++t) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 w4 = *(const float4*)&ws[t][4 * q];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float e = v[t / 3][k + t % 3];
          acc[k][4 * q] = fmaf(e, w4.x, acc[k][4 * q]);
          acc[k][4 * q + 1] = fmaf(e, w4.y, acc[k][4 * q + 1]);
          acc[k][4 * q + 2] = fmaf(e, w4.z, acc[k][4 * q + 2]);
          acc[k][4 * q + 3] = fmaf(e, w4.w, acc[k][4 * q + 3]);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      __align__(16) bf16 o[16];
#pragma unroll
      for (int c = 0; c < 16; ++c)
        o[c] = __float2bfloat16(relu ? fmaxf(acc[k][c], 0.f) : acc[k][c]);
      bf16* dst = (bf16*)out.p + (ny * W + x0 + k) * out.ps + out.off;
      *(uint4*)dst = *(const uint4*)o;
      *(uint4*)(dst + 8) = *(const uint4*)(o + 8);
    }
  }
}

// The inputs of the weight- and input-gradient kernels of a layer: the FP32
// gradient of its output, masked by its ReLU (act > 0), rounded to BF16 into a
// dense [pixels][C] buffer.  Where the gradient comes straight from another
// layer's input-gradient convolution, that kernel's epilogue writes it; these two
// form it from what arrives through an upsampling and through a skip connection
// and a pooling.  Eight channels per thread (C, strides and offsets multiples
// of 8).
__device__ __forceinline__ void gz_store(const float* v, Tensor act, long long p, int c, bf16* out,
                                         int C) {
  __align__(16) bf16 m[8], o[8];
  *(uint4*)m = *(const uint4*)((const bf16*)act.p + p * act.ps + act.off + c);
#pragma unroll
  for (int j = 0; j < 8; ++j)
    o[j] = __float2bfloat16(__bfloat162float(m[j]) <= 0.f ? 0.f : v[j]);
  *(uint4*)(out + p * C + c) = *(const uint4*)o;
}
__device__ __forceinline__ void ld8(const Tensor& t, long long p, int c, float* v) {
  const float4* q = (const float4*)((const float*)t.p + p * t.ps + t.off + c);
  const float4 a = q[0], b = q[1];
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

// transpose of the nearest 2x upsampling (the sum of the four output pixels)
__global__ void __launch_bounds__(256) k_up_bwd_gz(Tensor gout, Tensor act, bf16* out, int N, int H,
                                                   int W, int C) {   // H, W: input (low-res) sizes
  const int C8 = C / 8;
  const long long total = (long long)N * H * W * C8;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % C8) * 8;
    const long long p = i / C8;
    const int x = (int)(p % W);
    const long long ny = p / W;
    const long long q0 = (2 * ny) * (2 * W) + 2 * x;
    float g[4][8], s[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) ld8(gout, q0 + (k >> 1) * 2 * W + (k & 1), c, g[k]);
#pragma unroll
    for (int j = 0; j < 8; ++j) s[j] = ((g[0][j] + g[1][j]) + g[2][j]) + g[3][j];
    gz_store(s, act, p, c, out, C);
  }
}

// gradient of a pooled skip connection: g plus a quarter of the pooled map's
__global__ void __launch_bounds__(256) k_pool_bwd_gz(Tensor g, Tensor gpool, Tensor act, bf16* out,
                                                     int N, int H, int W, int C) {
  const int C8 = C / 8;
  const long long total = (long long)N * H * W * C8;   // H, W: full-resolution sizes
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % C8) * 8;
    const long long p = i / C8;
    const int x = (int)(p % W);
    const long long ny = p / W;                 // n * H + y, H even
    float v[8], q[8];
    ld8(g, p, c, v);
    ld8(gpool, (ny / 2) * (W / 2) + x / 2, c, q);
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = fmaf(0.25f, q[j], v[j]);
    gz_store(v, act, p, c, out, C);
  }
}

// The head's backward in one pass over the outputs: with y, t planar [N][C][P]
// (P pixels) and a = the head's BF16 input [N P][16],
//   loss += sum_c lam_c mean (y - t)^2,   gy = its derivative (FP32, not stored),
//   gz[p][:] = BF16 of the masked input gradient sum_c gy[p][c] w[c][:] (a > 0),
//   gw[c][:] += sum_p gy[p][c] a[p][:],   gb[c] += sum_p gy[p][c],
// all in FP32 but the loss, which is summed in FP64: its squares leave FP32's range from
// differences of 1.8e19 on (and below 1e-19).  A CTA takes tiles of 128 pixels (one per
// thread) and, along the grid's y, 32 output channels for gw; the y = 0 CTAs also form
// gz.  gy and the tile's inputs meet in shared memory, where each warp adds its 32
// pixels to its own copy of gw: lane (ci, half) owns channels half, half + 2, ..  What
// bounds it is HBM (y, t and the 16-channel maps once) and the FP64 units (a conversion,
// a product and a multiply-add per output): 8 images 256 x 1024, 25 channels, a whole
// training step 4.93 ms with the loss in pairs of FP32, 5.05 ms so (5.16 ms with lam
// converted for every output).
// WS: the head's weights (FP32) are in shared memory; else (very many channels) read
// from global memory.
constexpr int kHeadPix = 128, kHeadCh = 32, kHeadMaxShared = 1024;
template <bool WS>
__global__ void __launch_bounds__(kHeadPix) k_head_bwd(const float* __restrict__ y,
                                                       const float* __restrict__ t,
                                                       const float* __restrict__ lam,
                                                       const bf16* __restrict__ a,
                                                       const bf16* __restrict__ w, bf16* gz,
                                                       float* gw, float* gb, long long P, int C,
                                                       int N, double* loss) {
  constexpr int LD = kHeadPix + 4;
  __shared__ __align__(16) float gys[kHeadCh][LD];
  __shared__ __align__(16) float as[16][LD];
  __shared__ double red[kHeadPix / 32];
  extern __shared__ __align__(16) float wsh[];   // the head's weights [C][16], then lam [C] in FP64
  double* const lsh = (double*)(wsh + C * 16);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (WS)
    for (int i = tid; i < C * 16; i += kHeadPix) wsh[i] = __bfloat162float(w[i]);
  if (WS)
    for (int i = tid; i < C; i += kHeadPix) lsh[i] = lam[i];
  const int cb = blockIdx.y * kHeadCh, ci = lane & 15, half = lane >> 4;
  const bool first = blockIdx.y == 0;
  const double inv = 1.0 / ((double)P * N);
  const float inv2 = (float)(2.0 * inv);
  float acc[kHeadCh / 2], bacc = 0.f;
#pragma unroll
  for (int k = 0; k < kHeadCh / 2; ++k) acc[k] = 0.f;
  for (int i = tid; i < kHeadCh * LD; i += kHeadPix) ((float*)gys)[i] = 0.f;   // channels >= C
  __syncthreads();
  double s = 0.0;                                // the loss, FP64 as its squares may leave FP32
  const long long total = P * N;
  for (long long t0 = blockIdx.x * (long long)kHeadPix; t0 < total;
       t0 += (long long)gridDim.x * kHeadPix) {
    const long long q = t0 + tid;
    const bool ok = q < total;
    const long long n = ok ? q / P : 0, p = ok ? q - n * P : 0;
    float av[16], gd[16];
    {
      __align__(16) bf16 m[16];
      *(uint4*)m = ok ? *(const uint4*)(a + q * 16) : make_uint4(0u, 0u, 0u, 0u);
      *(uint4*)(m + 8) = ok ? *(const uint4*)(a + q * 16 + 8) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        av[j] = __bfloat162float(m[j]);
        as[j][tid] = av[j];
        gd[j] = 0.f;
      }
    }
    const float* yp = y + n * C * P + p;
    const float* tp = t + n * C * P + p;
    const int c0 = first ? 0 : cb, c1 = first ? C : min(C, cb + kHeadCh);
    for (int cc = c0; cc < c1; cc += 8) {       // eight channels' loads in flight
      float yv[8], tv[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const bool in = ok && cc + k < c1;
        yv[k] = in ? __ldg(yp + (long long)(cc + k) * P) : 0.f;
        tv[k] = in ? __ldg(tp + (long long)(cc + k) * P) : 0.f;
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int c = cc + k;
        if (c >= c1) break;
        const float l = __ldg(lam + c), e = yv[k] - tv[k];
        const float g = inv2 * l * e;
        if (c >= cb && c < cb + kHeadCh) gys[c - cb][tid] = g;
        if (first) {
          const double e64 = e;
          s = fma((WS ? lsh[c] : (double)l) * e64, e64, s);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            float4 wv;
            if (WS) {
              wv = *(const float4*)(wsh + c * 16 + 4 * j);
            } else {
              const bf16* wg = w + c * 16 + 4 * j;
              wv = make_float4(__bfloat162float(wg[0]), __bfloat162float(wg[1]),
                               __bfloat162float(wg[2]), __bfloat162float(wg[3]));
            }
            gd[4 * j] = fmaf(g, wv.x, gd[4 * j]);
            gd[4 * j + 1] = fmaf(g, wv.y, gd[4 * j + 1]);
            gd[4 * j + 2] = fmaf(g, wv.z, gd[4 * j + 2]);
            gd[4 * j + 3] = fmaf(g, wv.w, gd[4 * j + 3]);
          }
        }
      }
    }
    if (first && ok) {
      __align__(16) bf16 o[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) o[j] = __float2bfloat16(av[j] <= 0.f ? 0.f : gd[j]);
      *(uint4*)(gz + q * 16) = *(const uint4*)o;
      *(uint4*)(gz + q * 16 + 8) = *(const uint4*)(o + 8);
    }
    __syncwarp();
    // the warp's own 32 pixels (its lanes wrote them)
#pragma unroll 2
    for (int px = warp * 32; px < warp * 32 + 32; px += 4) {
      const float4 d = *(const float4*)&as[ci][px];
#pragma unroll
      for (int k = 0; k < kHeadCh / 2; ++k) {
        const float4 g = *(const float4*)&gys[2 * k + half][px];
        acc[k] = fmaf(g.x, d.x, fmaf(g.y, d.y, fmaf(g.z, d.z, fmaf(g.w, d.w, acc[k]))));
      }
    }
#pragma unroll
    for (int px = warp * 32; px < warp * 32 + 32; px += 4) {
      const float4 g = *(const float4*)&gys[lane][px];
      bacc += (g.x + g.y) + (g.z + g.w);
    }
    __syncwarp();
  }
  // the warps' sums, then one atomic per weight and CTA
  __syncthreads();
  float* sum = &gys[0][0];                       // [kHeadCh][17]
  for (int v = 0; v < kHeadPix / 32; ++v) {
    if (warp == v) {
#pragma unroll
      for (int k = 0; k < kHeadCh / 2; ++k) {
        float* d = sum + (2 * k + half) * 17 + ci;
        *d = v == 0 ? acc[k] : *d + acc[k];
      }
      float* d = sum + lane * 17 + 16;
      *d = v == 0 ? bacc : *d + bacc;
    }
    __syncthreads();
  }
  for (int i = tid; i < kHeadCh * 17; i += kHeadPix) {
    const int c = cb + i / 17, j = i % 17;
    if (c < C) atomicAdd(j < 16 ? gw + c * 16 + j : gb + c, sum[i]);
  }
  if (!first) return;
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) red[warp] = s;
  __syncthreads();
  if (tid == 0) {
    for (int i = 1; i < kHeadPix / 32; ++i) s += red[i];
    atomicAdd(loss, s * inv);
  }
}

// Weight and bias gradients of the first layer (one input channel, FP32): with
// x the BF16 image and g the FP32 gradient of the layer's 16 outputs masked by
// its ReLU, gw[co][tap] += sum_p g[p][co] x[p + tap].  Thread (pixel, half of the
// channels) keeps 8 x 9 sums in registers; a CTA adds them over shared memory and
// leaves one atomic per weight.  Bound by HBM (the gradient and the mask once).
__global__ void __launch_bounds__(256) k_wgrad_first(const bf16* __restrict__ x, Tensor g, Tensor act,
                                                     float* gw, float* gb, int N, int H, int W) {
  __shared__ float red[8][2][80];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, h = tid & 1;
  float acc[8][9], bs[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    bs[j] = 0.f;
#pragma unroll
    for (int k = 0; k < 9; ++k) acc[j][k] = 0.f;
  }
  const long long total = (long long)N * H * W;
  for (long long p = blockIdx.x * 128LL + (tid >> 1); p < total; p += gridDim.x * 128LL) {
    const int xx = (int)(p % W);
    const long long ny = p / W;
    const int yy = (int)(ny % H);
    float v[8], xv[9];
    ld8(g, p, 8 * h, v);
    __align__(16) bf16 m[8];
    *(uint4*)m = *(const uint4*)((const bf16*)act.p + p * act.ps + act.off + 8 * h);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const int y1 = yy + k / 3 - 1, x1 = xx + k % 3 - 1;
      xv[k] = (y1 >= 0 && y1 < H && x1 >= 0 && x1 < W)
                  ? __bfloat162float(x[p + (long long)(k / 3 - 1) * W + (k % 3 - 1)]) : 0.f;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float gj = __bfloat162float(m[j]) <= 0.f ? 0.f : v[j];
      bs[j] += gj;
#pragma unroll
      for (int k = 0; k < 9; ++k) acc[j][k] = fmaf(xv[k], gj, acc[j][k]);
    }
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {
#pragma unroll
    for (int k = 0; k < 10; ++k) {
      float r = k < 9 ? acc[j][k] : bs[j];
      for (int o = 16; o > 1; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
      if (lane < 2) red[warp][lane][j * 10 + k] = r;
    }
  }
  __syncthreads();
  if (tid < 160) {
    const int hh = tid / 80, e = tid % 80, co = 8 * hh + e / 10, k = e % 10;
    float r = 0.f;
    for (int w = 0; w < 8; ++w) r += red[w][hh][e];
    atomicAdd(k < 9 ? gw + co * 9 + k : gb + co, r);
  }
}

// Adam on the flat FP32 master parameters
__global__ void k_adam(float* w, const float* g, float* m, float* v, long long n, float lr,
                       float b1, float b2, float eps, float c1, float c2) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// The BF16 copies of a layer's FP32 OIHW master weights that its kernels read
// (null where none does): wf [tap][ci][co] (first layer), wt [tap][co][ci] with the
// taps flipped (head backward), wn [tap][co][ci] (the mma.sync head), and for the
// tcgen05 convolutions wp (forward) and wtp (input gradient: channels exchanged, taps
// flipped) in the order in which they lie in shared memory, one contiguous block per
// output-channel tile and chunk of 16 input channels (see tc_weight).
struct WCopies {
  bf16 *wf = nullptr, *wt = nullptr, *wn = nullptr, *wp = nullptr, *wtp = nullptr;
  int nt_p = 0, nt_t = 0;       // output-channel tiles of wp and wtp
};
// [tile][chunk][tap][channel octet][NT outputs][8 inputs] of weight (out o, in i)
__host__ __device__ __forceinline__ long long tc_weight(int o, int i, int tap, int nch, int taps,
                                                        int NT) {
  return (((((long long)(o / NT) * nch + i / 16) * taps + tap) * 2 + (i / 8) % 2) * NT + o % NT) * 8 +
         i % 8;
}
__global__ void k_wconv(const float* w, WCopies c, int co_n, int ci_n, int K) {
  const int total = co_n * ci_n * K * K;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const int kx = i % K, ky = (i / K) % K, ci = (i / (K * K)) % ci_n, co = i / (K * K * ci_n);
    const int tap = ky * K + kx, tapf = (K * K - 1) - tap;
    const bf16 b = __float2bfloat16(w[i]);
    if (c.wf) c.wf[((long long)tap * ci_n + ci) * co_n + co] = b;
    if (c.wt) c.wt[((long long)tapf * co_n + co) * ci_n + ci] = b;
    if (c.wn) c.wn[((long long)tap * co_n + co) * ci_n + ci] = b;
    if (c.wp) c.wp[tc_weight(co, ci, tap, ci_n / 16, K * K, c.nt_p)] = b;
    if (c.wtp) c.wtp[tc_weight(ci, co, tapf, co_n / 16, K * K, c.nt_t)] = b;
  }
}

// Output-channel tile of the tcgen05 convolution with `cout` outputs (0: none is
// compiled).
int tc_tile(int K, int cout) {
  const int nt = (cout + 15) / 16 * 16;
  if (K == 1) return nt <= 48 ? nt : 0;
  switch (nt) {
    case 16: return 16;
    case 48: case 144: return 48;
    case 64: return 64;
    case 96: case 288: return 96;
    case 192: return 192;
    default: return 0;
  }
}

__device__ __forceinline__ void ldsm_x4(uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3,
                                        const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"((unsigned)__cvta_generic_to_shared(p)));
}

__device__ __forceinline__ void mma_bf16(float* c, uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The head where it is wider than the tcgen05 tiles (mma.sync m16n8k16, BF16 operands,
// FP32 accumulation): out [pixels][Cout] = bias + in [pixels][16] w^T, w [Cout][16].  CTA:
// 128 pixels x 16 NB output channels, 8 warps of 16 pixels each, both operands staged in
// shared memory (rows padded by 8 elements against bank conflicts).
template <int NB>
__global__ void __launch_bounds__(256, 2) k_head_mma(const bf16* __restrict__ in,
                                                     const bf16* __restrict__ w,
                                                     const float* __restrict__ bias, float* out,
                                                     long long npix, int Cout) {
  constexpr int LD = 24, NT = NB * 16;
  __shared__ __align__(16) bf16 xs[128 * LD], ws[NT * LD];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long p0 = blockIdx.x * 128LL;
  const int co0 = blockIdx.y * NT;
  {
    const int v = tid & 1, px = tid >> 1;          // 16-byte vectors of 8 channels
    uint4 val = make_uint4(0u, 0u, 0u, 0u);
    if (p0 + px < npix) val = *(const uint4*)(in + (p0 + px) * 16 + 8 * v);
    *(uint4*)(xs + px * LD + 8 * v) = val;
  }
  for (int e = tid; e < NT * 2; e += 256) {
    const int v = e & 1, c = e >> 1;
    uint4 val = make_uint4(0u, 0u, 0u, 0u);
    if (co0 + c < Cout) val = *(const uint4*)(w + (co0 + c) * 16 + 8 * v);
    *(uint4*)(ws + c * LD + 8 * v) = val;
  }
  __syncthreads();
  float acc[2 * NB][4];
#pragma unroll
  for (int j = 0; j < 2 * NB; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
  uint32_t a0, a1, a2, a3;
  ldsm_x4(a0, a1, a2, a3, xs + (warp * 16 + (lane & 15)) * LD + ((lane >> 4) << 3));
#pragma unroll
  for (int nb = 0; nb < NB; ++nb) {
    uint32_t b0, b1, b2, b3;                       // two n8 blocks of 16 output channels
    const int bn = nb * 16 + (lane & 7) + ((lane >> 4) << 3), bk = ((lane >> 3) & 1) << 3;
    ldsm_x4(b0, b1, b2, b3, ws + bn * LD + bk);
    mma_bf16(acc[2 * nb], a0, a1, a2, a3, b0, b1);
    mma_bf16(acc[2 * nb + 1], a0, a1, a2, a3, b2, b3);
  }
  // c0, c1 at (pixel g, channels 2t, 2t+1), c2, c3 at pixel g + 8
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const long long p = p0 + warp * 16 + g + 8 * h;
    if (p >= npix) continue;
#pragma unroll
    for (int j = 0; j < 2 * NB; ++j) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int co = co0 + 8 * j + 2 * t + u;
        if (co < Cout) out[p * Cout + co] = acc[j][2 * h + u] + bias[co];
      }
    }
  }
}

// Training targets in normalised units from a solve's model m [N][C-1][P] and
// final residual weights wr [N][P]: t = m / rms, log(wr) - wr_pow log(rms).
__global__ void k_targets(const float* m, const float* wr, const float* rms, float* t,
                          long long P, int C, int N, float wr_pow) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < P * C * N;
       i += (long long)gridDim.x * blockDim.x) {
    const long long p = i % P;
    const int c = (int)((i / P) % C);
    const long long n = i / (P * C);
    const float r = rms[n];
    t[i] = (c < C - 1) ? m[(n * (C - 1) + c) * P + p] / r
                       : logf(fmaxf(wr[n * P + p], 1e-30f)) - wr_pow * logf(r);
  }
}

// -------------------------------------------------------------------------
struct Layer {
  int ci, co, k;
  long long w_off, b_off;   // into the flat parameter buffer
  WCopies c;
};

int grid1d(long long n) {
  long long b = (n + 255) / 256;
  return (int)(b > 152 * 16 ? 152 * 16 : (b < 1 ? 1 : b));
}

}  // namespace

using namespace ashrt;

struct ashrt_unet {
  int H = 0, W = 0, cout = 0, maxb = 0;
  int ch[4] = {16, 48, 96, 192};
  std::vector<Layer> L;              // 15 layers, reference order
  long long nparam = 0;
  float *w = nullptr, *g = nullptr, *am = nullptr, *av = nullptr;   // master, grad, Adam
  long long adam_t = 0;
  // activations (bf16) and gradients (fp32)
  std::vector<void*> allocs;
  bf16 *x, *e1a, *cat1, *p1, *e2a, *cat2, *p2, *e3a, *cat3, *p3, *ba, *bb, *d3a, *d3b, *d2a, *d2b,
      *d1a, *d1b;
  float *y, *ynhwc = nullptr, *g1a, *gcat1, *gp1, *gcat2, *gp2, *gcat3, *gp3;
  float *rms, *lam;
  double* rmsacc;
  bf16 *gza, *gzb;   // BF16 masked output gradients of two successive layers
  int* err;    // set by a tensor-core kernel whose bounded wait ran out
  double* loss;
  std::vector<float> lam_h;
};

namespace {

template <typename T>
cudaError_t dalloc(ashrt_unet* u, T** p, size_t n) {
  cudaError_t e = cudaMalloc((void**)p, n * sizeof(T) + 16);
  if (e == cudaSuccess) u->allocs.push_back(*p);
  return e;
}

Tensor T_(void* p, int ps, int off = 0) {
  Tensor t;
  t.p = p;
  t.ps = ps;
  t.off = off;
  return t;
}

// ---------------------------------------------------------------------------
// 5th-generation tensor-core (tcgen05) forward convolution.  M = 128 pixels of
// one image row (one TMEM lane each), N = the layer's output channels rounded
// up to 16 (one tile, <= 256 FP32 TMEM columns), K = 16 input channels per
// MMA, one MMA per tap, accumulated in TMEM over taps and channel chunks.
// Per 16-channel chunk the CTA stages, in the canonical K-major no-swizzle
// layout of 8-row x 16-byte core matrices,
//   A: [dy][2 channel octets][130 pixels][8 channels]  (a tap's A operand
//      starts dx pixels in: rows 16 B apart, next 8 pixels at +128 B = SBO,
//      next channel octet at +130 x 16 B = LBO)
//   B: [tap][2 octets][NT channels][8 input channels]  (SBO 128 B, LBO NT x 16 B),
// B once per CTA where all chunks' weights fit in 48 KB.
// One persistent CTA per SM walks over its tiles with three roles:
//   warps 8..11 copy (cp.async) the chunks of one tile after the other into a ring
//     of three to six stages, three chunks ahead of the one they hand over;
//   one thread of warp 12 issues the taps' MMAs of each chunk and commits them to
//     the stage's "empty" barrier, and a tile's last chunk to "tile done";
//   warps 0..7 read a finished tile's accumulators with tcgen05.ld (warps w and w + 4:
//     lanes 32 (w mod 4)..+31, alternate column groups), fuse bias, ReLU or the
//     mask and store, while the next tile accumulates in the other half of TMEM.
// Every wait is bounded; one that runs out ends its role, then the others', and
// sets the error flag.  What bounds a layer is not the MMAs (tensor pipe active 6 to
// 16 % of the time, 4 images: at 32 cycles to read a 4 KB A operand they need 420 us of 16
// images) nor any other pipe (none above half): long-scoreboard waits lead, and the
// operands of a chunk are some 1600 copies of 16 bytes per four rows from four warps.
// 16 images 256 x 1024, the thirteen 3x3 layers and the head: with one tile per
// CTA, two to three CTAs per SM and two stages the copies (800 us), MMAs (540) and
// stores (440) ran one after the other, 2190 us; so 1280 us.  Weights in their own
// order (32-byte pieces, the same ones for every SM at once) held the wide layers
// back: packed blocks took the 192-channel layers from 301 to 134 us.
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);   // version 1, no swizzle
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// Waits for the barrier phase; false after about a second.
__device__ __forceinline__ bool tc_wait(uint64_t* bar, uint32_t parity) {
  for (int i = 0; i < (1 << 22); ++i) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.b32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    if (i > 64) __nanosleep(256);
  }
  return false;
}

// Where a planar head output goes.  Channel c < C - 1 of image n: main + n
// main_n + c P; the last one: last + n last_n (either may be null).  With rms the
// outputs are returned in input units: the panels times rms[n], the last channel
// as exp(y) rms[n]^wr_pow.
struct HeadOut {
  float *main = nullptr, *last = nullptr;
  long long main_n = 0, last_n = 0;
  const float* rms = nullptr;
  float wr_pow = 0.f;
};

// Pixel-major head output [N][P][C] to its planar place: one thread per pixel.
__global__ void k_unpack_out(const float* y, HeadOut h, long long P, int C, int N) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < P * N;
       i += (long long)gridDim.x * blockDim.x) {
    const long long n = i / P, p = i % P;
    const float r = h.rms ? h.rms[n] : 1.f;
    const float* yi = y + i * C;
    if (h.main)
      for (int c = 0; c < C - 1; ++c) h.main[n * h.main_n + c * P + p] = h.rms ? yi[c] * r : yi[c];
    if (h.last)
      h.last[n * h.last_n + p] = h.rms ? expf(yi[C - 1]) * powf(r, h.wr_pow) : yi[C - 1];
  }
}

struct TcConvArgs {
  Tensor in;             // bf16 NHWC slice, ps and off multiples of 8
  const bf16* w;         // as they lie in shared memory (tc_weight)
  const float* bias;     // [Cout]
  Tensor out;            // bf16 or fp32 NHWC slice
  int N, H, W, Cin, Cout, relu;
  int* err;              // set to 1 if the MMA completion wait ran out
  int planar = 0;        // 1: planar FP32 output as in `head` (out unused)
  Tensor mask;           // BF16 activation: outputs where it is <= 0 are zeroed, or p == nullptr
  HeadOut head;          // planar: where the outputs go
};

// (L2::128B: a pixel's other channels, in the same line, are copied next)
__device__ __forceinline__ void cp16_line(void* dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global.L2::128B [%0], [%1], 16, %2;\n" ::"r"(smem_addr(dst)),
               "l"(src), "r"(valid ? 16 : 0)
               : "memory");
}

__device__ __forceinline__ void cp16(void* dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_addr(dst)), "l"(src),
               "r"(valid ? 16 : 0)
               : "memory");
}

template <int K, int NT, int RR>
struct TcTile {
  static constexpr int R = K / 2, PW = 128 + 2 * R, TAPS = K * K, ROWS = RR + 2 * R;
  static constexpr int DS = (NT + 31) / 32 * 32;        // TMEM columns per output row
  static constexpr int NCOL = RR * DS <= 32 ? 32 : RR * DS <= 64 ? 64 : RR * DS <= 128 ? 128 : 256;
  static constexpr uint32_t A_PLANE = PW * 16, B_PLANE = NT * 16;       // bytes per channel octet
  static constexpr uint32_t A_BYTES = ROWS * 2 * A_PLANE, B_BYTES = TAPS * 2 * B_PLANE;
  // the weights of all channel chunks stay in shared memory where they are small
  static bool resident(int nch) { return nch * B_BYTES <= 48 * 1024; }
  // stages of the ring in about 200 KB, three to six
  static int stages(int nch) {
    const bool res = resident(nch);
    const int n = (int)((205 * 1024 - (res ? nch * B_BYTES : 0)) / (A_BYTES + (res ? 0 : B_BYTES)));
    return n > 6 ? 6 : n;
  }
  // more than half an SM's, so that one CTA is resident (it holds up to all of TMEM)
  static size_t smem(int nch) {
    const size_t n = (size_t)stages(nch) * (A_BYTES + (resident(nch) ? 0 : B_BYTES)) +
                     (resident(nch) ? nch * B_BYTES : 0) + 256;
    return n < 120 * 1024 ? 120 * 1024 : n;
  }
};

constexpr int kTcEpi = 256, kTcCopy = 128, kTcThreads = kTcEpi + kTcCopy + 32;
constexpr int kTcAhead = 2;   // chunks copied beyond the one handed over (stages >= kTcAhead + 1)

__device__ __forceinline__ void tc_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
          smem_addr(bar))
      : "memory");
}

template <int K, int NT, int RR, typename TO>
__global__ void __launch_bounds__(kTcThreads, 1) k_conv_tc(TcConvArgs a, int n_tiles, int stages,
                                                           int b_resident) {
  using S = TcTile<K, NT, RR>;
  constexpr int R = S::R, TAPS = S::TAPS, ROWS = S::ROWS, DS = S::DS, NCOL = S::NCOL;
  constexpr uint32_t A_PLANE = S::A_PLANE, B_PLANE = S::B_PLANE;
  constexpr uint32_t A_BYTES = S::A_BYTES, B_BYTES = S::B_BYTES;
  static_assert(RR * DS <= 256, "TMEM tile");
  constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NT >> 3) << 17) |
                             ((uint32_t)(128 >> 4) << 24);        // F32 += BF16 x BF16, M 128
  extern __shared__ __align__(128) unsigned char smt[];
  const int nch = a.Cin / 16;
  unsigned char* const Bbase = smt + stages * A_BYTES;
  uint64_t* full = (uint64_t*)(Bbase + (b_resident ? nch : stages) * B_BYTES);
  uint64_t *empty = full + 6, *tfull = full + 12, *tempty = full + 14;
  uint32_t* tslot = (uint32_t*)(full + 16);
  __shared__ __align__(16) float sbias[NT];
  const int tid = threadIdx.x, warp = tid >> 5;
  const int xt = (a.W + 127) / 128, yt = (a.H + RR - 1) / RR;
  const int co0 = blockIdx.y * NT;                // output-channel tile
  if (tid < NT) sbias[tid] = a.bias && co0 + tid < a.Cout ? a.bias[co0 + tid] : 0.f;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_addr(tslot)),
                 "r"((uint32_t)(2 * NCOL)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (tid == 0) {
    for (int i = 0; i < 16; ++i)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(full + i)),
                   "r"(i < 6 ? kTcCopy : i < 14 ? 1 : kTcEpi));
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = *tslot;
  bool ok = true;

  if (warp >= kTcEpi / 32 && warp < (kTcEpi + kTcCopy) / 32) {
    // ---- copies: two threads per pixel, one 16-byte octet each (zero-filled
    // outside the image); the 2 R halo pixels at a row's end by the first threads
    const int t = tid - kTcEpi, sp = t >> 1, so = t & 1, hr = t >> 2, hp = 128 + (sp & 1);
    const bf16* in = (const bf16*)a.in.p;
    const long long rstride = (long long)a.W * a.in.ps;
    const uint4* wsrc = (const uint4*)a.w + (size_t)blockIdx.y * nch * (B_BYTES / 16);
    auto stage_b = [&](int c, unsigned char* Bs) {
      const uint4* src = wsrc + (size_t)c * (B_BYTES / 16);
#pragma unroll 6
      for (int e = t; e < (int)(B_BYTES / 16); e += kTcCopy) cp16(Bs + e * 16, src + e, true);
    };
    // hands over stage st: its copies are complete and visible to the MMAs
    auto hand_over = [&](int st) {
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      tc_arrive(full + st);
    };
    if (b_resident)
      for (int c = 0; c < nch; ++c) stage_b(c, Bbase + c * B_BYTES);
    int st = 0, out = 0, n = 0;              // stage of this step, of the next hand-over; steps
    uint32_t phase = 1;                      // parity the stage's previous use leaves
    for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
      const int x0 = (tile % xt) * 128 - R, rb = tile / xt, y0 = (rb % yt) * RR - R;
      const bf16* src = in + (((long long)(rb / yt) * a.H + y0) * a.W + x0) * a.in.ps + a.in.off + 8 * so;
      for (int c = 0; c < nch; ++c, src += 16, ++n) {
        if (!(ok = tc_wait(empty + st, phase))) break;
        unsigned char* As = smt + st * A_BYTES;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const int px = sp + 64 * half;
          const bool okx = x0 + px >= 0 && x0 + px < a.W;
          const bf16* s0 = src + (long long)px * a.in.ps;
#pragma unroll
          for (int r = 0; r < ROWS; ++r) {
            const bool in_img = okx && y0 + r >= 0 && y0 + r < a.H;
            cp16_line(As + (r * 2 + so) * A_PLANE + px * 16, in_img ? s0 + r * rstride : in, in_img);
          }
        }
        if (R > 0 && t < 4 * ROWS) {
          const bool in_img = x0 + hp < a.W && y0 + hr >= 0 && y0 + hr < a.H;
          cp16_line(As + (hr * 2 + so) * A_PLANE + hp * 16,
               in_img ? src + hr * rstride + (long long)hp * a.in.ps : in, in_img);
        }
        if (!b_resident) stage_b(c, Bbase + st * B_BYTES);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        if (n >= kTcAhead) {
          asm volatile("cp.async.wait_group %0;\n" ::"n"(kTcAhead) : "memory");
          hand_over(out);
          out = out + 1 == stages ? 0 : out + 1;
        }
        if (++st == stages) {
          st = 0;
          phase ^= 1u;
        }
      }
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    for (int i = n < kTcAhead ? n : kTcAhead; i > 0 && ok; --i) {
      hand_over(out);
      out = out + 1 == stages ? 0 : out + 1;
    }
  } else if (warp == (kTcEpi + kTcCopy) / 32) {
    // ---- MMAs: one thread
    if ((tid & 31) == 0) {
      int st = 0, k = 0;
      uint32_t phase = 0;
      for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x, ++k) {
        // the accumulators' previous tile has been read
        ok = tc_wait(tempty + (k & 1), ((k >> 1) & 1) ^ 1);
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        for (int c = 0; c < nch && ok; ++c) {
          if (!(ok = tc_wait(full + st, phase))) break;
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
          const uint32_t As = smem_addr(smt + st * A_BYTES);
          const uint32_t Bs = smem_addr(Bbase + (b_resident ? c : st) * B_BYTES);
#pragma unroll
          for (int r = 0; r < RR; ++r) {
#pragma unroll
            for (int tap = 0; tap < TAPS; ++tap) {
              const int dy = tap / K, dx = tap % K;
              const uint64_t ad = umma_desc(As + (r + dy) * 2 * A_PLANE + dx * 16, A_PLANE, 128);
              const uint64_t bd = umma_desc(Bs + tap * 2 * B_PLANE, B_PLANE, 128);
              const uint32_t acc = (c > 0 || tap > 0) ? 1u : 0u;
              asm volatile(
                  "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                  " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
                      tmem + (uint32_t)((k & 1) * NCOL + r * DS)),
                  "l"(ad), "l"(bd), "r"(IDESC), "r"(acc));
            }
          }
          tc_commit(empty + st);
          if (c + 1 == nch) tc_commit(tfull + (k & 1));
          if (++st == stages) {
            st = 0;
            phase ^= 1u;
          }
        }
      }
    }
  } else {
    int k = 0;
    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++k) {
      const int x0 = (tile % xt) * 128, rb = tile / xt, n = rb / yt, y0 = (rb % yt) * RR;
      const uint32_t tacc = tmem + (uint32_t)((k & 1) * NCOL);
      ok = tc_wait(tfull + (k & 1), (k >> 1) & 1);
      if (!__all_sync(0xffffffffu, ok)) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      // epilogue: thread = pixel (TMEM lane of its warp quarter); warps w and
      // w + 4 share lanes and split the (row, 16-column) groups
      const int lane_base = (warp & 3) * 32;
      const int xx = x0 + lane_base + (tid & 31);
      TO* out = (TO*)a.out.p;
      constexpr int G = NT / 16;
      for (int gi = warp >> 2; gi < RR * G; gi += 2) {
        const int r = gi / G, c0 = (gi % G) * 16;
        uint32_t v[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
            "%11, %12, %13, %14, %15}, [%16];\n"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
              "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
              "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
            : "r"(tacc + ((uint32_t)lane_base << 16) + (uint32_t)(r * DS + c0)));
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
        const int y = y0 + r;
        if (xx < a.W && y < a.H) {
          const long long pix = ((long long)n * a.H + y) * a.W + xx;
          const int cb = co0 + c0;                    // first output channel of the group
          float f[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            f[j] = __uint_as_float(v[j]) + sbias[c0 + j];
            if (a.relu) f[j] = fmaxf(f[j], 0.f);
          }
          const bool whole = cb + 16 <= a.Cout;
          if (a.planar) {
            // the stores of a warp are contiguous
            const long long P = (long long)a.H * a.W, p = (long long)y * a.W + xx;
            const float rms = a.head.rms ? a.head.rms[n] : 1.f;
            float* o = a.head.main ? a.head.main + n * a.head.main_n + cb * P + p : nullptr;
            float flast = 0.f;
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              if (o && cb + j < a.Cout - 1) o[j * P] = a.head.rms ? f[j] * rms : f[j];
              flast = cb + j == a.Cout - 1 ? f[j] : flast;
            }
            if (a.head.last && cb < a.Cout && cb + 16 >= a.Cout)
              a.head.last[n * a.head.last_n + p] =
                  a.head.rms ? expf(flast) * powf(rms, a.head.wr_pow) : flast;
          } else if (sizeof(TO) == 2 && whole && ((a.out.ps | a.out.off) & 7) == 0) {
            __align__(16) bf16 o[16];
            if (a.mask.p) {
              const uint4* mp = (const uint4*)((const bf16*)a.mask.p + pix * a.mask.ps + a.mask.off + cb);
              __align__(16) bf16 m[16];
              *(uint4*)m = mp[0];
              *(uint4*)(m + 8) = mp[1];
#pragma unroll
              for (int j = 0; j < 16; ++j)
                if (__bfloat162float(m[j]) <= 0.f) f[j] = 0.f;
            }
#pragma unroll
            for (int j = 0; j < 16; ++j) o[j] = __float2bfloat16(f[j]);
            bf16* dst = (bf16*)out + pix * a.out.ps + a.out.off + cb;
            *(uint4*)dst = *(const uint4*)o;
            *(uint4*)(dst + 8) = *(const uint4*)(o + 8);
          } else if (sizeof(TO) == 4 && whole && ((a.out.ps | a.out.off) & 3) == 0) {
            float4* dst = (float4*)((float*)out + pix * a.out.ps + a.out.off + cb);
#pragma unroll
            for (int q = 0; q < 4; ++q) dst[q] = make_float4(f[4 * q], f[4 * q + 1], f[4 * q + 2], f[4 * q + 3]);
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (cb + j < a.Cout) st_f(out, pix * a.out.ps + a.out.off + cb + j, f[j]);
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      tc_arrive(tempty + (k & 1));
    }
  }
  if (!ok && a.err) atomicExch(a.err, 1);
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"((uint32_t)(2 * NCOL)));
  }
}

template <int K, int NT, int RR, typename TO>
void conv_tc_v(const TcConvArgs& a, cudaStream_t s) {
  using S = TcTile<K, NT, RR>;
  const int nch = a.Cin / 16;
  const size_t smem = S::smem(nch);
  static SmemAttr attr;
  set_smem(k_conv_tc<K, NT, RR, TO>, smem, attr);
  const int tiles = a.N * ((a.H + RR - 1) / RR) * ((a.W + 127) / 128);
  const int gy = (a.Cout + NT - 1) / NT;
  const int gx = std::min(tiles, std::max(1, 152 / gy));   // one CTA per SM
  k_conv_tc<K, NT, RR, TO><<<dim3(gx, gy), kTcThreads, smem, s>>>(a, tiles, S::stages(nch),
                                                                 S::resident(nch) ? 1 : 0);
  count_launches(1);
}

// tcgen05 forward convolution for the layer sizes of the network; false if the
// output-channel tile is not one of the compiled ones (the caller then uses
// the mma.sync kernel)
template <int K, typename TO>
bool conv_tc(Tensor in, const bf16* w, const float* bias, Tensor out, int N, int H, int W,
             int Cin, int Cout, int relu, int* err, cudaStream_t s, int planar = 0,
             Tensor mask = Tensor(), HeadOut head = HeadOut()) {
  if (Cin % 16 != 0 || in.ps % 8 != 0 || in.off % 8 != 0) return false;
  TcConvArgs a;
  a.planar = planar;
  a.mask = mask;
  a.head = head;
  a.in = in;
  a.w = w;
  a.bias = bias;
  a.out = out;
  a.N = N;
  a.H = H;
  a.W = W;
  a.Cin = Cin;
  a.Cout = Cout;
  a.relu = relu;
  a.err = err;
  if constexpr (K == 3) {
    // output rows per CTA: the staged input rows serve RR outputs (TMEM:
    // RR x NT <= 256); wider outputs are split into NT-channel tiles
    switch (tc_tile(K, Cout)) {
      case 16: conv_tc_v<3, 16, 4, TO>(a, s); return true;
      case 48: conv_tc_v<3, 48, 4, TO>(a, s); return true;
      case 64: conv_tc_v<3, 64, 4, TO>(a, s); return true;
      case 96: conv_tc_v<3, 96, 2, TO>(a, s); return true;
      case 192: conv_tc_v<3, 192, 1, TO>(a, s); return true;
      default: return false;
    }
  } else {
    switch (tc_tile(K, Cout)) {
      case 16: conv_tc_v<1, 16, 4, TO>(a, s); return true;
      case 32: conv_tc_v<1, 32, 4, TO>(a, s); return true;
      case 48: conv_tc_v<1, 48, 4, TO>(a, s); return true;
      default: return false;
    }
  }
}

// The wide head (more than 48 channels): the widest tile that divides its channels.
template <int NB>
void head_mma_v(const bf16* in, const bf16* w, const float* bias, float* out, long long npix,
                int Cout, cudaStream_t s) {
  const dim3 grid((unsigned)((npix + 127) / 128), (Cout + NB * 16 - 1) / (NB * 16));
  k_head_mma<NB><<<grid, 256, 0, s>>>(in, w, bias, out, npix, Cout);
  count_launches(1);
}
void head_mma(const bf16* in, const bf16* w, const float* bias, float* out, long long npix, int Cout,
              cudaStream_t s) {
  if (Cout % 64 == 0) head_mma_v<4>(in, w, bias, out, npix, Cout, s);
  else if (Cout % 48 == 0) head_mma_v<3>(in, w, bias, out, npix, Cout, s);
  else if (Cout % 32 == 0) head_mma_v<2>(in, w, bias, out, npix, Cout, s);
  else head_mma_v<4>(in, w, bias, out, npix, Cout, s);
}

// rms[g] of the n input gathers x [n][per]
void compute_rms(ashrt_unet* u, const float* x, long long per, int n, cudaStream_t s) {
  cudaMemsetAsync(u->rmsacc, 0, sizeof(double) * n, s);
  k_sumsq<<<dim3(64, n), 256, 0, s>>>(x, per, u->rmsacc);
  k_rms_fin<<<(n + 127) / 128, 128, 0, s>>>(u->rmsacc, per, u->rms, n);
  count_launches(2);
}

// Planar outputs [n][cout][P] at y.
HeadOut head_planar(const ashrt_unet* u, float* y) {
  HeadOut h;
  const long long P = (long long)u->H * u->W;
  h.main = y;
  h.last = y + (u->cout - 1) * P;
  h.main_n = h.last_n = u->cout * P;
  return h;
}

// Forward pass on `n` images already packed in u->x; the head's output goes where
// `head` says.
void net_forward(ashrt_unet* u, int n, cudaStream_t s, const HeadOut& head) {
  const int H = u->H, W = u->W, c0 = u->ch[0], c1 = u->ch[1], c2 = u->ch[2], c3 = u->ch[3];
  const Tensor none = T_(nullptr, 0);
  auto& L = u->L;
  auto B = [&](int i) { return u->w + L[i].b_off; };
  auto grid = [&](long long cnt) { return grid1d(cnt); };
  // encoder
  k_conv_first<<<grid((long long)n * H * W / 4), 256, 0, s>>>(u->x, L[0].c.wf, B(0), T_(u->e1a, c0), n,
                                                          H, W, 1);
  conv_tc<3, bf16>(T_(u->e1a, c0), L[1].c.wp, B(1), T_(u->cat1, c1 + c0, c1), n, H, W, c0, c0, 1, u->err, s);
  k_pool<<<grid((long long)n * H * W / 4 * c0 / 8), 256, 0, s>>>(T_(u->cat1, c1 + c0, c1), T_(u->p1, c0), n, H, W, c0);
  conv_tc<3, bf16>(T_(u->p1, c0), L[2].c.wp, B(2), T_(u->e2a, c1), n, H / 2, W / 2, c0, c1, 1, u->err, s);
  conv_tc<3, bf16>(T_(u->e2a, c1), L[3].c.wp, B(3), T_(u->cat2, c2 + c1, c2), n, H / 2, W / 2, c1, c1, 1, u->err, s);
  k_pool<<<grid((long long)n * H * W / 16 * c1 / 8), 256, 0, s>>>(T_(u->cat2, c2 + c1, c2), T_(u->p2, c1), n, H / 2, W / 2, c1);
  conv_tc<3, bf16>(T_(u->p2, c1), L[4].c.wp, B(4), T_(u->e3a, c2), n, H / 4, W / 4, c1, c2, 1, u->err, s);
  conv_tc<3, bf16>(T_(u->e3a, c2), L[5].c.wp, B(5), T_(u->cat3, c3 + c2, c3), n, H / 4, W / 4, c2, c2, 1, u->err, s);
  k_pool<<<grid((long long)n * H * W / 64 * c2 / 8), 256, 0, s>>>(T_(u->cat3, c3 + c2, c3), T_(u->p3, c2), n, H / 4, W / 4, c2);
  conv_tc<3, bf16>(T_(u->p3, c2), L[6].c.wp, B(6), T_(u->ba, c3), n, H / 8, W / 8, c2, c3, 1, u->err, s);
  conv_tc<3, bf16>(T_(u->ba, c3), L[7].c.wp, B(7), T_(u->bb, c3), n, H / 8, W / 8, c3, c3, 1, u->err, s);
  // decoder
  k_up<<<grid((long long)n * H * W / 16 * c3 / 8), 256, 0, s>>>(T_(u->bb, c3), T_(u->cat3, c3 + c2, 0), n, H / 4, W / 4, c3);
  conv_tc<3, bf16>(T_(u->cat3, c3 + c2), L[8].c.wp, B(8), T_(u->d3a, c2), n, H / 4, W / 4, c3 + c2, c2, 1, u->err, s);
  conv_tc<3, bf16>(T_(u->d3a, c2), L[9].c.wp, B(9), T_(u->d3b, c2), n, H / 4, W / 4, c2, c2, 1, u->err, s);
  k_up<<<grid((long long)n * H * W / 4 * c2 / 8), 256, 0, s>>>(T_(u->d3b, c2), T_(u->cat2, c2 + c1, 0), n, H / 2, W / 2, c2);
  conv_tc<3, bf16>(T_(u->cat2, c2 + c1), L[10].c.wp, B(10), T_(u->d2a, c1), n, H / 2, W / 2, c2 + c1, c1, 1, u->err, s);
  conv_tc<3, bf16>(T_(u->d2a, c1), L[11].c.wp, B(11), T_(u->d2b, c1), n, H / 2, W / 2, c1, c1, 1, u->err, s);
  k_up<<<grid((long long)n * H * W * c1 / 8), 256, 0, s>>>(T_(u->d2b, c1), T_(u->cat1, c1 + c0, 0), n, H, W, c1);
  conv_tc<3, bf16>(T_(u->cat1, c1 + c0), L[12].c.wp, B(12), T_(u->d1a, c0), n, H, W, c1 + c0, c0, 1, u->err, s);
  conv_tc<3, bf16>(T_(u->d1a, c0), L[13].c.wp, B(13), T_(u->d1b, c0), n, H, W, c0, c0, 1, u->err, s);
  if (!conv_tc<1, float>(T_(u->d1b, c0), L[14].c.wp, B(14), none, n, H, W, c0, u->cout, 0, u->err, s, 1,
                         none, head)) {
    // a head wider than the tcgen05 tiles: pixel-major, then to its planar place
    const long long P = (long long)H * W;
    head_mma(u->d1b, L[14].c.wn, B(14), u->ynhwc, P * n, u->cout, s);
    k_unpack_out<<<grid1d(P * n), 256, 0, s>>>(u->ynhwc, head, P, u->cout, n);
    count_launches(1);
  }
  count_launches(7);   // pools, upsamplings, first layer
}

// Weight and bias gradients of a 3x3 layer on the tensor cores (mma.sync
// m16n8k16, BF16 operands, FP32 accumulation): for every tap, an implicit GEMM
// gw[co][ci] += sum_p gz[p][co] x[p + tap][ci] over the pixels p, M = output
// channels, N = input channels, K = pixels.  A CTA has nine warps, one per tap,
// owns 16 MT output x 8 NT input channels and reduces a 128-pixel column strip of
// rows_per image rows.  The input rows live in a ring of four: a row of output
// gradients [128][16 MT] needs three of them, of which two are there already,
// and the fourth is in flight with the next row of gradients, so every input row
// is copied once and no copy is waited for.  Both operands stay in their NHWC
// order and are read with ldmatrix.trans (row pitches of an odd number of 16-byte
// units: no bank conflicts); a tap that looks across the image's first or last
// row is left out for that row.  The
// tensor core's FP32 accumulation truncates, so its error grows with the length of a
// chain (584 steps of 16 pixels left 1.7e-5 of a gradient's norm, 216 a third of
// it): after `chain` rows a sum moves on, to a second set of registers where a tile
// has them to spare, with an atomic each otherwise.  CTAs of the first
// input-channel tile also sum the bias gradient.
// Channel tiles of 48 x 48 (the network's channels are multiples of 48 but for
// 16 and 64) waste nothing where 32 x 32 computed a third to a half of padding.
// 8 images 256 x 1024, all thirteen layers: 2.86 ms with a wait per row and no
// ring, 1.69 ms so, of which the shorter chains take 0.24.
struct WgMmaArgs {
  Tensor in;            // bf16 layer input slice (ps, off multiples of 8)
  const bf16* gz;       // bf16 masked output gradient, dense [pixels][Cout]
  float* gw;            // [Cout][Cin][3][3] fp32, accumulated
  float* gb;            // [Cout] fp32, accumulated
  int N, H, W, Cin, Cout, rows_per;
  int chain;            // image rows summed in one chain of the tensor core's accumulators
};

__device__ __forceinline__ void ldsm_x4_t(uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3,
                                          const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"((unsigned)__cvta_generic_to_shared(p)));
}

template <int MT, int NT>
__global__ void __launch_bounds__(288, MT * NT >= 18 ? 2 : 3) k_wgrad_mma(WgMmaArgs a) {
  constexpr int CO_T = 16 * MT, CI_T = 8 * NT, LDX = CI_T + 8, LDG = CO_T + 8, PW = 130, T = 288;
  constexpr int PARTS = T / CO_T;               // bias: threads per output channel
  extern __shared__ __align__(16) unsigned char smw[];
  bf16* xs = (bf16*)smw;                        // [4 rows][PW][LDX]
  bf16* gs = xs + 4 * PW * LDX;                 // [2 rows][128][LDG]
  const int tid = threadIdx.x, tap = tid >> 5, lane = tid & 31, dy = tap / 3, dx = tap % 3;
  const int xt = (a.W + 127) / 128;
  const int x0 = (blockIdx.x % xt) * 128;
  const int rows = a.N * a.H, row0 = (blockIdx.x / xt) * a.rows_per;
  const int row1 = min(row0 + a.rows_per, rows);
  const int ci0 = blockIdx.y * CI_T, co0 = blockIdx.z * CO_T;
  const bf16* in = (const bf16*)a.in.p;
  // input row R (over all images) into its place in the ring, and a row of output
  // gradients: two threads per pixel with adjacent 16-byte octets (one 32-byte
  // sector), the octets in steps of two
  const int sp = tid >> 1, so = (tid & 1) * 8;
  const bool okx = sp < PW && x0 + sp >= 1 && x0 + sp - 1 < a.W, okg = x0 + sp < a.W;
  const bf16* srcx = in + (long long)(x0 + sp - 1) * a.in.ps + a.in.off + ci0 + so;
  const bf16* srcg = a.gz + (long long)(x0 + sp) * a.Cout + co0 + so;
  auto load_x = [&](int R) {
    if (R < 0 || R >= rows || sp >= PW) return;   // (only taps that are left out would read R)
    bf16* dst = xs + ((R & 3) * PW + sp) * LDX + so;
    const bf16* src = srcx + (long long)R * a.W * a.in.ps;
#pragma unroll
    for (int q = 0; q < NT / 2; ++q) {
      const bool ok = okx && ci0 + 16 * q < a.Cin;
      cp16(dst + 16 * q, ok ? src + 16 * q : in, ok);
    }
  };
  auto load_g = [&](int R) {
    if (sp >= 128) return;
    bf16* dst = gs + ((R & 1) * 128 + sp) * LDG + so;
    const bf16* src = srcg + (long long)R * a.W * a.Cout;
#pragma unroll
    for (int q = 0; q < MT; ++q) {
      const bool ok = okg && co0 + 16 * q < a.Cout;
      cp16(dst + 16 * q, ok ? src + 16 * q : a.gz, ok);
    }
  };
  float acc[MT][NT][4];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j) acc[i][j][0] = acc[i][j][1] = acc[i][j][2] = acc[i][j][3] = 0.f;
  float bsum = 0.f;
  const bool bias = blockIdx.y == 0 && tid < PARTS * CO_T;
  constexpr bool TWO = MT * NT <= 6;            // registers for the sums of several chains
  float sum[MT][NT][4];   // (unused and so without registers otherwise)
  if (TWO) {
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
      for (int j = 0; j < NT; ++j) sum[i][j][0] = sum[i][j][1] = sum[i][j][2] = sum[i][j][3] = 0.f;
  }
  auto to_memory = [&](const float (&v)[MT][NT][4]) {
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int co = co0 + i * 16 + g + 8 * (e >> 1), ci = ci0 + j * 8 + 2 * t + (e & 1);
          if (co < a.Cout && ci < a.Cin)
            atomicAdd(&a.gw[((long long)co * a.Cin + ci) * 9 + tap], v[i][j][e]);
        }
  };
  int left = a.chain;

  load_x(row0 - 1);
  load_x(row0);
  load_x(row0 + 1);
  load_g(row0);
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  for (int row = row0; row < row1; ++row) {
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();   // this row's operands are there; the previous row's reads are done
    if (row + 1 < row1) {
      load_x(row + 2);
      load_g(row + 1);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    const bf16* g = gs + (row & 1) * 128 * LDG;
    if (bias)
      for (int px = tid / CO_T; px < 128; px += PARTS)
        bsum += __bfloat162float(g[px * LDG + tid % CO_T]);
    if (left-- == 0) {   // the chain ends: its sum moves on, rounded to nearest
      left = a.chain - 1;
      if (!TWO) to_memory(acc);
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if (TWO) sum[i][j][e] += acc[i][j][e];
            acc[i][j][e] = 0.f;
          }
    }
    const int y = row % a.H;
    if ((dy == 0 && y == 0) || (dy == 2 && y == a.H - 1)) continue;
    const bf16* x = xs + ((row + dy - 1) & 3) * PW * LDX + dx * LDX;
    const int kr = lane & 7, id = lane >> 3;
#pragma unroll 2
    for (int kb = 0; kb < 128; kb += 16) {
      uint32_t af[MT][4];
#pragma unroll
      for (int i = 0; i < MT; ++i)
        ldsm_x4_t(af[i][0], af[i][1], af[i][2], af[i][3],
                  g + (kb + kr + ((id >> 1) << 3)) * LDG + i * 16 + ((id & 1) << 3));
#pragma unroll
      for (int j = 0; j < NT; j += 2) {
        uint32_t b0, b1, b2, b3;
        ldsm_x4_t(b0, b1, b2, b3, x + (kb + kr + ((id & 1) << 3)) * LDX + (j + (id >> 1)) * 8);
#pragma unroll
        for (int i = 0; i < MT; ++i) {
          mma_bf16(acc[i][j], af[i][0], af[i][1], af[i][2], af[i][3], b0, b1);
          mma_bf16(acc[i][j + 1], af[i][0], af[i][1], af[i][2], af[i][3], b2, b3);
        }
      }
    }
  }
  if (TWO) {
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[i][j][e] += sum[i][j][e];
  }
  to_memory(acc);
  if (bias && co0 + tid % CO_T < a.Cout) atomicAdd(&a.gb[co0 + tid % CO_T], bsum);
}

template <int MT, int NT>
void wgrad_mma_v(const WgMmaArgs& a0, cudaStream_t s) {
  WgMmaArgs a = a0;
  constexpr size_t smem = (size_t)(4 * 130 * (8 * NT + 8) + 2 * 128 * (16 * MT + 8)) * sizeof(bf16);
  static SmemAttr attr;
  set_smem(k_wgrad_mma<MT, NT>, smem, attr);
  const int xt = (a.W + 127) / 128;
  const unsigned gy = (a.Cin + 8 * NT - 1) / (8 * NT), gz = (a.Cout + 16 * MT - 1) / (16 * MT);
  // one wave of two or three CTAs per SM: each extra strip costs its atomics again
  const int res = MT * NT >= 18 ? 2 : 3;
  const long long rows = (long long)a.N * a.H, want = 152LL * res / ((long long)gy * gz * xt);
  const long long per_col = std::max(1LL, std::min(want, rows));
  a.rows_per = (int)((rows + per_col - 1) / per_col);
  // rows to a chain: as many as give about 152 x 8 chains in all per 32 x 32 channels
  // (32 x 16 for 16 output channels)
  const long long tiles = (long long)((a.Cin + 31) / 32) * (a.Cout <= 16 ? 1 : (a.Cout + 31) / 32);
  const long long chains = std::min(rows, ((152LL * 8 + tiles - 1) / tiles + xt - 1) / xt);
  a.chain = (int)((rows + chains - 1) / chains);
  const long long nstrip = (rows + a.rows_per - 1) / a.rows_per;
  k_wgrad_mma<MT, NT><<<dim3((unsigned)(nstrip * xt), gy, gz), 288, smem, s>>>(a);
  count_launches(1);
}

// Backward of 3x3 layer l (input `in`, BF16 masked output gradient gz): weight
// and bias gradients, and the input gradient either as FP32 into `out` or, with
// `act` (the ReLU output that is the layer's input), masked and rounded into
// gz_out for the layer before.
void layer_backward(ashrt_unet* u, Tensor in, const bf16* gz, const Layer& l, Tensor out,
                    Tensor act, bf16* gz_out, int n, int H, int W, cudaStream_t s) {
  WgMmaArgs a;
  a.in = in;
  a.gz = gz;
  a.gw = u->g + l.w_off;
  a.gb = u->g + l.b_off;
  a.N = n;
  a.H = H;
  a.W = W;
  a.Cin = l.ci;
  a.Cout = l.co;
  // channel tiles 16 MT x 8 NT: the widest that divides both channel counts
  if (l.co % 48 == 0) {
    if (l.ci % 48 == 0) wgrad_mma_v<3, 6>(a, s);
    else wgrad_mma_v<3, 2>(a, s);
  } else {
    if (l.ci % 32 == 0) wgrad_mma_v<1, 4>(a, s);
    else wgrad_mma_v<1, 2>(a, s);
  }
  const Tensor g = T_(const_cast<bf16*>(gz), l.co);
  if (gz_out)
    conv_tc<3, bf16>(g, l.c.wtp, nullptr, T_(gz_out, l.ci), n, H, W, l.co, l.ci, 0, u->err, s, 0, act);
  else
    conv_tc<3, float>(g, l.c.wtp, nullptr, out, n, H, W, l.co, l.ci, 0, u->err, s);
}

// Backward pass from the planar head output u->y and the targets; accumulates
// parameter gradients in u->g and the loss in u->loss.
void net_backward(ashrt_unet* u, const float* target, int n, cudaStream_t s) {
  const int H = u->H, W = u->W, c0 = u->ch[0], c1 = u->ch[1], c2 = u->ch[2], c3 = u->ch[3];
  const Tensor none = T_(nullptr, 0);
  auto& L = u->L;
  auto grid = [&](long long cnt) { return grid1d(cnt); };
  bf16 *ga = u->gza, *gb = u->gzb;   // masked output gradients of a layer and of the one before
  const long long P = (long long)H * W;
  const dim3 hg((unsigned)std::min<long long>((P * n + kHeadPix - 1) / kHeadPix, 152 * 8),
                (u->cout + kHeadCh - 1) / kHeadCh);
  const bool ws = u->cout <= kHeadMaxShared;
  const size_t head_ch = 16 * sizeof(float) + sizeof(double), hs = ws ? u->cout * head_ch : 0;
  auto* head = ws ? k_head_bwd<true> : k_head_bwd<false>;
  // (beside 26 KB of static shared memory; few heads are this wide: set on every call)
  if (hs > 16 * 1024)
    cudaFuncSetAttribute(head, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(kHeadMaxShared * head_ch));
  head<<<hg, kHeadPix, hs, s>>>(u->y, target, u->lam, u->d1b, L[14].c.wt, ga,
                                u->g + L[14].w_off, u->g + L[14].b_off, P, u->cout, n, u->loss);
  // dec1
  layer_backward(u, T_(u->d1a, c0), ga, L[13], none, T_(u->d1a, c0), gb, n, H, W, s);
  layer_backward(u, T_(u->cat1, c1 + c0), gb, L[12], T_(u->gcat1, c1 + c0), none, nullptr, n, H, W, s);
  k_up_bwd_gz<<<grid(P * n / 4 * c1 / 8), 256, 0, s>>>(T_(u->gcat1, c1 + c0, 0), T_(u->d2b, c1), ga,
                                                       n, H / 2, W / 2, c1);
  // dec2
  layer_backward(u, T_(u->d2a, c1), ga, L[11], none, T_(u->d2a, c1), gb, n, H / 2, W / 2, s);
  layer_backward(u, T_(u->cat2, c2 + c1), gb, L[10], T_(u->gcat2, c2 + c1), none, nullptr, n, H / 2,
                 W / 2, s);
  k_up_bwd_gz<<<grid(P * n / 16 * c2 / 8), 256, 0, s>>>(T_(u->gcat2, c2 + c1, 0), T_(u->d3b, c2), ga,
                                                        n, H / 4, W / 4, c2);
  // dec3
  layer_backward(u, T_(u->d3a, c2), ga, L[9], none, T_(u->d3a, c2), gb, n, H / 4, W / 4, s);
  layer_backward(u, T_(u->cat3, c3 + c2), gb, L[8], T_(u->gcat3, c3 + c2), none, nullptr, n, H / 4,
                 W / 4, s);
  k_up_bwd_gz<<<grid(P * n / 64 * c3 / 8), 256, 0, s>>>(T_(u->gcat3, c3 + c2, 0), T_(u->bb, c3), ga,
                                                        n, H / 8, W / 8, c3);
  // bottleneck
  layer_backward(u, T_(u->ba, c3), ga, L[7], none, T_(u->ba, c3), gb, n, H / 8, W / 8, s);
  layer_backward(u, T_(u->p3, c2), gb, L[6], T_(u->gp3, c2), none, nullptr, n, H / 8, W / 8, s);
  // enc3 (its output s3 lives in cat3[c3:], gradient in gcat3[c3:])
  k_pool_bwd_gz<<<grid(P * n / 16 * c2 / 8), 256, 0, s>>>(T_(u->gcat3, c3 + c2, c3), T_(u->gp3, c2),
                                                          T_(u->cat3, c3 + c2, c3), ga, n, H / 4,
                                                          W / 4, c2);
  layer_backward(u, T_(u->e3a, c2), ga, L[5], none, T_(u->e3a, c2), gb, n, H / 4, W / 4, s);
  layer_backward(u, T_(u->p2, c1), gb, L[4], T_(u->gp2, c1), none, nullptr, n, H / 4, W / 4, s);
  // enc2
  k_pool_bwd_gz<<<grid(P * n / 4 * c1 / 8), 256, 0, s>>>(T_(u->gcat2, c2 + c1, c2), T_(u->gp2, c1),
                                                         T_(u->cat2, c2 + c1, c2), ga, n, H / 2,
                                                         W / 2, c1);
  layer_backward(u, T_(u->e2a, c1), ga, L[3], none, T_(u->e2a, c1), gb, n, H / 2, W / 2, s);
  layer_backward(u, T_(u->p1, c0), gb, L[2], T_(u->gp1, c0), none, nullptr, n, H / 2, W / 2, s);
  // enc1: the first layer's gradients are FP32 throughout
  k_pool_bwd_gz<<<grid(P * n * c0 / 8), 256, 0, s>>>(T_(u->gcat1, c1 + c0, c1), T_(u->gp1, c0),
                                                     T_(u->cat1, c1 + c0, c1), ga, n, H, W, c0);
  layer_backward(u, T_(u->e1a, c0), ga, L[1], T_(u->g1a, c0), none, nullptr, n, H, W, s);
  k_wgrad_first<<<(unsigned)std::min<long long>((P * n + 127) / 128, 152 * 3), 256, 0, s>>>(
      u->x, T_(u->g1a, c0), T_(u->e1a, c0), u->g + L[0].w_off, u->g + L[0].b_off, n, H, W);
  count_launches(8);
}

cudaError_t refresh_bf16_weights(ashrt_unet* u, cudaStream_t s) {
  for (auto& l : u->L) {
    const int total = l.co * l.ci * l.k * l.k;
    k_wconv<<<(total + 255) / 256, 256, 0, s>>>(u->w + l.w_off, l.c, l.co, l.ci, l.k);
    count_launches(1);
  }
  return cudaGetLastError();
}

}  // namespace

extern "C" {

ashrt_status ashrt_unet_create(ashrt_unet** out, int H, int W, int out_channels, int max_batch,
                               const float* init_params, long long n_init) {
  if (!out || H < 8 || W < 8 || H % 8 || W % 8 || out_channels < 1 || max_batch < 1) {
    set_error("ashrt_unet_create: need H, W multiples of 8 (>= 8), out_channels >= 1, max_batch >= 1");
    return ASHRT_EINVAL;
  }
  *out = nullptr;
  ashrt_unet* u = new ashrt_unet();
  u->H = H;
  u->W = W;
  u->cout = out_channels;
  u->maxb = max_batch;
  const int c0 = u->ch[0], c1 = u->ch[1], c2 = u->ch[2], c3 = u->ch[3];
  const int spec[15][3] = {{1, c0, 3},       {c0, c0, 3},      {c0, c1, 3}, {c1, c1, 3},
                           {c1, c2, 3},      {c2, c2, 3},      {c2, c3, 3}, {c3, c3, 3},
                           {c3 + c2, c2, 3}, {c2, c2, 3},      {c2 + c1, c1, 3}, {c1, c1, 3},
                           {c1 + c0, c0, 3}, {c0, c0, 3},      {c0, out_channels, 1}};
  long long off = 0;
  for (auto& sp : spec) {
    Layer l;
    l.ci = sp[0];
    l.co = sp[1];
    l.k = sp[2];
    l.w_off = off;
    off += (long long)l.co * l.ci * l.k * l.k;
    l.b_off = off;
    off += l.co;
    u->L.push_back(l);
  }
  u->nparam = off;
  const long long P0 = (long long)max_batch * H * W;
  cudaError_t e = cudaSuccess;
  auto A = [&](auto** p, size_t n) {
    if (e == cudaSuccess) e = dalloc(u, p, n);
  };
  A(&u->w, off);
  A(&u->g, off);
  A(&u->am, off);
  A(&u->av, off);
  for (auto& l : u->L) {
    const size_t n = (size_t)l.co * l.ci * l.k * l.k;
    const bool first = &l == &u->L.front();
    if (first) A(&l.c.wf, n);
    if (l.k == 1) {
      A(&l.c.wt, n);
      if (!tc_tile(1, l.co)) A(&l.c.wn, n);
    }
    if (!first && (l.c.nt_p = tc_tile(l.k, l.co))) {
      // a head of any width fills whole tiles (zeros)
      const size_t np = n / l.co * ((l.co + l.c.nt_p - 1) / l.c.nt_p * l.c.nt_p);
      A(&l.c.wp, np);
      if (e == cudaSuccess) e = cudaMemset(l.c.wp, 0, np * sizeof(bf16));
    }
    if (!first && l.k == 3) {
      l.c.nt_t = tc_tile(3, l.ci);
      A(&l.c.wtp, n);
    }
  }
  A(&u->x, P0);
  A(&u->e1a, P0 * c0);
  A(&u->cat1, P0 * (c1 + c0));
  A(&u->p1, P0 / 4 * c0);
  A(&u->e2a, P0 / 4 * c1);
  A(&u->cat2, P0 / 4 * (c2 + c1));
  A(&u->p2, P0 / 16 * c1);
  A(&u->e3a, P0 / 16 * c2);
  A(&u->cat3, P0 / 16 * (c3 + c2));
  A(&u->p3, P0 / 64 * c2);
  A(&u->ba, P0 / 64 * c3);
  A(&u->bb, P0 / 64 * c3);
  A(&u->d3a, P0 / 16 * c2);
  A(&u->d3b, P0 / 16 * c2);
  A(&u->d2a, P0 / 4 * c1);
  A(&u->d2b, P0 / 4 * c1);
  A(&u->d1a, P0 * c0);
  A(&u->d1b, P0 * c0);
  A(&u->y, P0 * out_channels);
  if (out_channels > 48) A(&u->ynhwc, P0 * out_channels);   // head not on the tcgen05 kernel
  A(&u->g1a, P0 * c0);
  A(&u->gcat1, P0 * (c1 + c0));
  A(&u->gp1, P0 / 4 * c0);
  A(&u->gcat2, P0 / 4 * (c2 + c1));
  A(&u->gp2, P0 / 16 * c1);
  A(&u->gcat3, P0 / 16 * (c3 + c2));
  A(&u->gp3, P0 / 64 * c2);
  A(&u->rms, max_batch);
  A(&u->rmsacc, max_batch);
  A(&u->gza, P0 * c0);
  A(&u->gzb, P0 * c0);
  A(&u->err, 1);
  A(&u->lam, out_channels);
  A(&u->loss, 1);
  if (e != cudaSuccess) {
    cudaGetLastError();
    set_error("ashrt_unet_create: cudaMalloc failed: %s", cudaGetErrorString(e));
    for (void* p : u->allocs) cudaFree(p);
    delete u;
    return ASHRT_ENOMEM;
  }
  // parameters: given, or He-normal from a fixed-seed generator (host, Box-Muller)
  std::vector<float> h(off, 0.f);
  if (init_params) {
    if (n_init != off) {
      set_error("ashrt_unet_create: %lld initial parameters given, the network has %lld", n_init, off);
      for (void* p : u->allocs) cudaFree(p);
      delete u;
      return ASHRT_EINVAL;
    }
    for (long long i = 0; i < off; ++i) h[i] = init_params[i];
  } else {
    uint64_t st = 0x9e3779b97f4a7c15ull;
    auto uni = [&]() {
      st ^= st << 13;
      st ^= st >> 7;
      st ^= st << 17;
      return ((st >> 11) + 0.5) * (1.0 / 9007199254740992.0);
    };
    for (auto& l : u->L) {
      const double sd = std::sqrt(2.0 / (l.ci * l.k * l.k));
      for (long long i = 0; i < (long long)l.co * l.ci * l.k * l.k; ++i) {
        const double a = uni(), b = uni();
        h[l.w_off + i] = (float)(sd * std::sqrt(-2.0 * std::log(a)) * std::cos(6.283185307179586 * b));
      }
    }
  }
  e = cudaMemcpy(u->w, h.data(), off * 4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(u->am, 0, off * 4);
  if (e == cudaSuccess) e = cudaMemset(u->err, 0, sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(u->av, 0, off * 4);
  if (e == cudaSuccess) e = cudaMemset(u->g, 0, off * 4);
  if (e == cudaSuccess) e = refresh_bf16_weights(u, 0);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    set_error("ashrt_unet_create: init failed: %s", cudaGetErrorString(e));
    for (void* p : u->allocs) cudaFree(p);
    delete u;
    return ASHRT_ECUDA;
  }
  u->lam_h.assign(out_channels, 1.f);
  cudaMemcpy(u->lam, u->lam_h.data(), out_channels * 4, cudaMemcpyHostToDevice);
  *out = u;
  return ASHRT_OK;
}

void ashrt_unet_destroy(ashrt_unet* u) {
  if (!u) return;
  cudaDeviceSynchronize();
  for (void* p : u->allocs) cudaFree(p);
  delete u;
}

long long ashrt_unet_param_count(const ashrt_unet* u) { return u ? u->nparam : 0; }

ashrt_status ashrt_unet_get(const ashrt_unet* u, float* params, float* grads, long long n) {
  if (!u || n != u->nparam) {
    set_error("ashrt_unet_get: NULL network or wrong count");
    return ASHRT_EINVAL;
  }
  cudaError_t e = cudaDeviceSynchronize();
  int err = 0;
  if (e == cudaSuccess) e = cudaMemcpy(&err, u->err, sizeof(int), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && err) {
    cudaMemset(u->err, 0, sizeof(int));
    set_error("ashrt_unet_get: a tensor-core kernel's bounded wait ran out in an earlier call");
    return ASHRT_ETIMEOUT;
  }
  if (e == cudaSuccess && params) e = cudaMemcpy(params, u->w, n * 4, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && grads) e = cudaMemcpy(grads, u->g, n * 4, cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) {
    set_error("ashrt_unet_get: %s", cudaGetErrorString(e));
    return ASHRT_ECUDA;
  }
  return ASHRT_OK;
}

// x: [n][H][W] fp32 inputs (gathers [nx][nt]); y: [n][cout][H][W] fp32 outputs.
// Inputs are scaled by their RMS; with `rescale` the outputs are returned in
// input units for an IRLS misfit power p: channels < cout-1 multiplied by the
// RMS (model panels), the last channel as exp(y) * RMS^((p-2)/2) (residual
// weights).
ashrt_status ashrt_unet_forward(ashrt_unet* u, const float* x, float* y, int n, int rescale,
                                float p, void* stream) {
  if (!u || !x || !y || n < 1 || n > u->maxb) {
    set_error("ashrt_unet_forward: NULL argument or n outside [1, max_batch]");
    return ASHRT_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const long long per = (long long)u->H * u->W;
  compute_rms(u, x, per, n, s);
  k_pack_in<<<grid1d(per * n), 256, 0, s>>>(x, u->rms, u->x, per, n);
  count_launches(1);
  HeadOut head = head_planar(u, y);
  if (rescale) {
    head.rms = u->rms;
    head.wr_pow = 0.5f * (p - 2.f);
  }
  net_forward(u, n, s, head);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error("ashrt_unet_forward: %s", cudaGetErrorString(e));
    return ASHRT_ECUDA;
  }
  return ASHRT_OK;
}

// One training step on n pairs: x [n][H][W], target [n][cout][H][W] (targets
// in the network's normalised units), per-channel loss weights (host, cout
// values, or NULL = 1).  Adam with the given learning rate; returns the loss.
ashrt_status ashrt_unet_train_step(ashrt_unet* u, const float* x, const float* target, int n,
                                   const float* channel_weight, float lr, double* loss_out,
                                   void* stream) {
  if (!u || !x || !target || n < 1 || n > u->maxb) {
    set_error("ashrt_unet_train_step: NULL argument or n outside [1, max_batch]");
    return ASHRT_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const long long per = (long long)u->H * u->W;
  if (channel_weight) {
    bool same = true;
    for (int c = 0; c < u->cout; ++c) same = same && (u->lam_h[c] == channel_weight[c]);
    if (!same) {
      u->lam_h.assign(channel_weight, channel_weight + u->cout);
      cudaMemcpyAsync(u->lam, u->lam_h.data(), u->cout * 4, cudaMemcpyHostToDevice, s);
    }
  }
  cudaMemsetAsync(u->loss, 0, sizeof(double), s);
  cudaMemsetAsync(u->g, 0, u->nparam * 4, s);
  compute_rms(u, x, per, n, s);
  k_pack_in<<<grid1d(per * n), 256, 0, s>>>(x, u->rms, u->x, per, n);
  count_launches(1);
  net_forward(u, n, s, head_planar(u, u->y));
  net_backward(u, target, n, s);
  if (lr > 0.f) {
    u->adam_t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - std::pow(b1, (float)u->adam_t);
    const float c2 = 1.f - std::pow(b2, (float)u->adam_t);
    k_adam<<<grid1d(u->nparam), 256, 0, s>>>(u->w, u->g, u->am, u->av, u->nparam, lr, b1, b2,
                                            1e-8f, c1, c2);
    count_launches(1);
    refresh_bf16_weights(u, s);
  }
  cudaError_t e = cudaGetLastError();
  int err = 0;
  if (e == cudaSuccess && loss_out) {
    e = cudaMemcpyAsync(loss_out, u->loss, sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&err, u->err, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  }
  if (e != cudaSuccess) {
    set_error("ashrt_unet_train_step: %s", cudaGetErrorString(e));
    return ASHRT_ECUDA;
  }
  if (err) {
    cudaMemsetAsync(u->err, 0, sizeof(int), s);
    set_error("ashrt_unet_train_step: a tensor-core kernel's bounded wait ran out");
    return ASHRT_ETIMEOUT;
  }
  return ASHRT_OK;
}

ashrt_status ashrt_unet_targets(ashrt_unet* u, const float* x, const float* m, const float* wr,
                                float* t, int n, float p, void* stream) {
  if (!u || !x || !m || !wr || !t || n < 1 || n > u->maxb) {
    set_error("ashrt_unet_targets: NULL argument or n outside [1, max_batch]");
    return ASHRT_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const long long per = (long long)u->H * u->W;
  compute_rms(u, x, per, n, s);
  k_targets<<<grid1d(per * u->cout * n), 256, 0, s>>>(m, wr, u->rms, t, per, u->cout, n,
                                                      0.5f * (p - 2.f));
  count_launches(1);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error("ashrt_unet_targets: %s", cudaGetErrorString(e));
    return ASHRT_ECUDA;
  }
  return ASHRT_OK;
}

ashrt_status ashrt_unet_predict(ashrt_unet* u, const float* x, float* m0, float* wr0, int n,
                                float p, void* stream) {
  if (!u || !x || (!m0 && !wr0) || n < 1 || n > u->maxb) {
    set_error("ashrt_unet_predict: NULL argument or n outside [1, max_batch]");
    return ASHRT_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const long long per = (long long)u->H * u->W;
  compute_rms(u, x, per, n, s);
  k_pack_in<<<grid1d(per * n), 256, 0, s>>>(x, u->rms, u->x, per, n);
  count_launches(1);
  HeadOut head;
  head.main = m0;
  head.main_n = (u->cout - 1) * per;
  head.last = wr0;
  head.last_n = per;
  head.rms = u->rms;
  head.wr_pow = 0.5f * (p - 2.f);
  net_forward(u, n, s, head);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error("ashrt_unet_predict: %s", cudaGetErrorString(e));
    return ASHRT_ECUDA;
  }
  return ASHRT_OK;
}

}  // extern "C"

