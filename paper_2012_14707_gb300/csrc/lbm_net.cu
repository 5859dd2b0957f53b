// Warm-start network of liblbm.so (lbm_net_*): a 4-level convolutional
// encoder-decoder that predicts (rho, u) of a steady state from (solid
// mask, signed distance, Kn), trained on the GPU by the kernels below.
// The paper has no network; this is the learned initial state of the
// solver, which then runs to the same residual as from rest.
//
// Layout: activations NHWC, weights [kh][kw][ci][co] (the layout of the
// FP64 reference in the tests).  Activations and activation gradients are
// stored in BF16 (training) or FP32 (gradient checks); every
// product is accumulated in FP32; master weights, weight gradients and Adam
// moments are FP32.
//
// FP32 mode, on CUDA cores:
//   conv_fwd<KS>    y = act(conv(x, w) + b), KS = 3 (zero padding) or 1;
//                   a CTA computes a 16x16 pixel tile x 16 output channels,
//                   staging an input tile (with halo) and the weights of a
//                   16-channel input slice in shared memory.
//   conv_bwd_data   the same kernel on weights flipped in space and
//                   transposed in channels (a conv3x3 is its own adjoint
//                   pattern), after masking the output gradient by the ReLU.
//   conv_bwd_weight dW[dy][dx][c][o] = sum_pixels x[p + d][c] gz[p][o]: a
//                   CTA reduces a pixel chunk for a 16x16 (c, o) tile and
//                   adds it into FP32 dW; db by a column sum.
//   pool / upsample / concat / MSE / Adam: elementwise or simple reductions.
// BF16 mode: the convolutions of lbm_net_tc.cu on the tensor cores, which
// read the decoder's upsampled-and-concatenated input from its two sources
// and apply the ReLU's backward mask as they store, and elementwise passes
// of 8 channels per thread (below).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "../../include/lbm.h"
#include "lbm_internal.h"
#include "lbm_net_tc.h"

namespace lbm {
namespace net {
namespace {

constexpr int TP = 16;  // pixel tile edge
constexpr int TC = 16;  // channel tile (input slice and output block)

// y[n, i, j, o] = act(b[o] + sum x[n, i+dy-p, j+dx-p, c] w[dy][dx][c][o])
// over a channel range; `relu` applies max(., 0).  xs: channel stride of x
// (x may be a slice of a wider tensor: element (n,i,j,c) at
// ((n*H + i)*W + j)*xs + c).  Grid: (ceil(W/16)*ceil(H/16), ceil(Co/16), N).
template <int KS>
__global__ void __launch_bounds__(TP * TP)
conv_fwd(const float *__restrict__ x, int xs, const float *__restrict__ w,
         const float *__restrict__ b, float *__restrict__ y, int ys, int H, int W, int Ci, int Co,
         int relu) {
  constexpr int HALO = KS / 2;
  constexpr int T = TP + 2 * HALO;
  __shared__ float sx[T][T][TC + 1];  // +1: conflict-free strided reads
  __shared__ float sw[KS][KS][TC][TC];
  const int tiles_x = (W + TP - 1) / TP;
  const int ti = blockIdx.x / tiles_x, tj = blockIdx.x % tiles_x;
  const int o0 = blockIdx.y * TC;
  const int n = blockIdx.z;
  const int li = threadIdx.x / TP, lj = threadIdx.x % TP;
  const int i = ti * TP + li, j = tj * TP + lj;
  float acc[TC];
#pragma unroll
  for (int q = 0; q < TC; q++) acc[q] = 0.f;
  for (int c0 = 0; c0 < Ci; c0 += TC) {
    // input tile with halo
    for (int e = threadIdx.x; e < T * T * TC; e += TP * TP) {
      const int c = e % TC, p = e / TC, pj = p % T, pi = p / T;
      const int gi = ti * TP + pi - HALO, gj = tj * TP + pj - HALO;
      float v = 0.f;
      if (gi >= 0 && gi < H && gj >= 0 && gj < W && c0 + c < Ci)
        v = x[((static_cast<int64_t>(n) * H + gi) * W + gj) * xs + c0 + c];
      sx[pi][pj][c] = v;
    }
    for (int e = threadIdx.x; e < KS * KS * TC * TC; e += TP * TP) {
      const int o = e % TC, c = (e / TC) % TC, d = e / (TC * TC);
      float v = 0.f;
      if (c0 + c < Ci && o0 + o < Co) v = w[(static_cast<int64_t>(d) * Ci + c0 + c) * Co + o0 + o];
      sw[d / KS][d % KS][c][o] = v;
    }
    __syncthreads();
#pragma unroll
    for (int dy = 0; dy < KS; dy++)
#pragma unroll
      for (int dx = 0; dx < KS; dx++)
#pragma unroll 4
        for (int c = 0; c < TC; c++) {
          const float xv = sx[li + dy][lj + dx][c];
#pragma unroll
          for (int q = 0; q < TC; q++) acc[q] = fmaf(xv, sw[dy][dx][c][q], acc[q]);
        }
    __syncthreads();
  }
  if (i < H && j < W) {
    float *yp = y + ((static_cast<int64_t>(n) * H + i) * W + j) * ys;
#pragma unroll
    for (int q = 0; q < TC; q++) {
      if (o0 + q < Co) {
        float v = acc[q] + (b ? b[o0 + q] : 0.f);
        if (relu) v = fmaxf(v, 0.f);
        yp[o0 + q] = v;
      }
    }
  }
}

// dW[dy][dx][c][o] += sum over a pixel chunk of x[p + d - HALO][c] gz[p][o];
// db[o] += sum gz[p][o] (blockIdx.y == 0 tiles only).  Grid:
// (ceil(Ci/16) * ceil(Co/16), chunks); 256 threads = 16 (c) x 16 (o).
template <int KS>
__global__ void __launch_bounds__(256)
conv_bwd_weight(const float *__restrict__ x, int xs, const float *__restrict__ gz, int N, int H,
                int W, int Ci, int Co, int pix_per_chunk, float *__restrict__ dw,
                float *__restrict__ db) {
  constexpr int HALO = KS / 2;
  const int tiles_o = (Co + TC - 1) / TC;
  const int c0 = (blockIdx.x / tiles_o) * TC, o0 = (blockIdx.x % tiles_o) * TC;
  const int c = threadIdx.x / TC, o = threadIdx.x % TC;
  const int64_t npix = static_cast<int64_t>(N) * H * W;
  const int64_t p0 = static_cast<int64_t>(blockIdx.y) * pix_per_chunk;
  const int64_t p1 = p0 + pix_per_chunk < npix ? p0 + pix_per_chunk : npix;
  __shared__ float sg[32][TC];
  __shared__ float sxv[32][KS * KS][TC];
  float acc[KS * KS];
#pragma unroll
  for (int d = 0; d < KS * KS; d++) acc[d] = 0.f;
  float bacc = 0.f;
  for (int64_t pb = p0; pb < p1; pb += 32) {
    // stage 32 pixels: gz[p][o0..] and x[p + d][c0..] for every offset d
    for (int e = threadIdx.x; e < 32 * TC; e += 256) {
      const int pp = e / TC, oo = e % TC;
      const int64_t p = pb + pp;
      sg[pp][oo] = (p < p1 && o0 + oo < Co) ? gz[p * Co + o0 + oo] : 0.f;
    }
    for (int e = threadIdx.x; e < 32 * KS * KS * TC; e += 256) {
      const int cc = e % TC, d = (e / TC) % (KS * KS), pp = e / (TC * KS * KS);
      const int64_t p = pb + pp;
      float v = 0.f;
      if (p < p1 && c0 + cc < Ci) {
        const int64_t n = p / (static_cast<int64_t>(H) * W);
        const int rem = static_cast<int>(p - n * H * W);
        const int i = rem / W + d / KS - HALO, j = rem % W + d % KS - HALO;
        if (i >= 0 && i < H && j >= 0 && j < W)
          v = x[((n * H + i) * W + j) * xs + c0 + cc];
      }
      sxv[pp][d][cc] = v;
    }
    __syncthreads();
#pragma unroll 4
    for (int pp = 0; pp < 32; pp++) {
      const float g = sg[pp][o];
#pragma unroll
      for (int d = 0; d < KS * KS; d++) acc[d] = fmaf(sxv[pp][d][c], g, acc[d]);
      bacc += g;
    }
    __syncthreads();
  }
  if (c0 + c < Ci && o0 + o < Co) {
#pragma unroll
    for (int d = 0; d < KS * KS; d++)
      atomicAdd(&dw[(static_cast<int64_t>(d) * Ci + c0 + c) * Co + o0 + o], acc[d]);
    if (c == 0 && c0 == 0 && db) atomicAdd(&db[o0 + o], bacc);
  }
}

// wt[d'][o][c] = w[KS*KS-1-d'][c][o]: the weights of the adjoint convolution.
__global__ void flip_weights(const float *__restrict__ w, float *__restrict__ wt, int KS2, int Ci,
                             int Co) {
  const int64_t n = static_cast<int64_t>(KS2) * Ci * Co;
  for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < n;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int c = static_cast<int>(e % Ci), o = static_cast<int>((e / Ci) % Co),
              d = static_cast<int>(e / (static_cast<int64_t>(Ci) * Co));
    wt[e] = w[(static_cast<int64_t>(KS2 - 1 - d) * Ci + c) * Co + o];
  }
}

__global__ void to_storage(const float *__restrict__ s, float *__restrict__ d, int64_t n) {
  for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < n;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x)
    d[e] = s[e];
}

__global__ void to_float(const float *__restrict__ s, int ss, float *__restrict__ d, int C,
                         int64_t npix) {
  for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < npix * C;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t p = e / C;
    d[e] = s[p * ss + e % C];
  }
}

// g[p][c] *= (h[p][c] > 0)  (ReLU backward; h is the layer output)
__global__ void relu_mask(float *__restrict__ g, const float *__restrict__ h, int64_t n) {
  for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < n;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x)
    if (!(h[e] > 0.f)) g[e] = 0.f;
}

// 2x2 average pooling, y has H/2 x W/2 pixels; x channel stride xs.
__global__ void pool2_fwd(const float *__restrict__ x, int xs, float *__restrict__ y, int N, int H,
                          int W, int C) {
  const int h2 = H / 2, w2 = W / 2;
  const int64_t n_out = static_cast<int64_t>(N) * h2 * w2 * C;
  for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < n_out;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int c = static_cast<int>(e % C);
    const int64_t p = e / C;
    const int j = static_cast<int>(p % w2), i = static_cast<int>((p / w2) % h2);
    const int64_t n = p / (static_cast<int64_t>(w2) * h2);
    float s = 0.f;
    for (int a = 0; a < 2; a++)
      for (int bb = 0; bb < 2; bb++)
        s += x[((n * H + 2 * i + a) * W + 2 * j + bb) * xs + c];
    y[e] = 0.25f * s;
  }
}

// gx[.] (+)= gy / 4 spread over each 2x2 block; gx channel stride xs
__global__ void pool2_bwd(const float *__restrict__ gy, float *__restrict__ gx, int xs, int N,
                          int H, int W, int C, int accumulate) {
  const int64_t n_in = static_cast<int64_t>(N) * H * W * C;
  for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < n_in;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int c = static_cast<int>(e % C);
    const int64_t p = e / C;
    const int j = static_cast<int>(p % W), i = static_cast<int>((p / W) % H);
    const int64_t n = p / (static_cast<int64_t>(W) * H);
    float v = 0.25f * gy[((n * (H / 2) + i / 2) * (W / 2) + j / 2) * C + c];
    float *dst = gx + p * xs + c;
    if (accumulate) v += *dst;
    *dst = v;
  }
}

// y (channel stride ys, first C channels) = nearest 2x upsampling of x
__global__ void up2_fwd(const float *__restrict__ x, float *__restrict__ y, int ys, int N, int H,
                        int W, int C) {
  const int64_t n_out = static_cast<int64_t>(N) * H * W * C;  // H, W: output size
  for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < n_out;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int c = static_cast<int>(e % C);
    const int64_t p = e / C;
    const int j = static_cast<int>(p % W), i = static_cast<int>((p / W) % H);
    const int64_t n = p / (static_cast<int64_t>(W) * H);
    y[p * ys + c] = x[((n * (H / 2) + i / 2) * (W / 2) + j / 2) * C + c];
  }
}

// gx (H/2 x W/2, C channels) = sum of gy over each 2x2 block; gy channel stride gs
__global__ void up2_bwd(const float *__restrict__ gy, int gs, float *__restrict__ gx, int N, int H,
                        int W, int C) {
  const int h2 = H / 2, w2 = W / 2;
  const int64_t n_out = static_cast<int64_t>(N) * h2 * w2 * C;
  for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < n_out;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int c = static_cast<int>(e % C);
    const int64_t p = e / C;
    const int j = static_cast<int>(p % w2), i = static_cast<int>((p / w2) % h2);
    const int64_t n = p / (static_cast<int64_t>(w2) * h2);
    float s = 0.f;
    for (int a = 0; a < 2; a++)
      for (int bb = 0; bb < 2; bb++) s += gy[((n * H + 2 * i + a) * W + 2 * j + bb) * gs + c];
    gx[e] = s;
  }
}

// copy C channels between tensors with channel strides (and offsets applied by the caller)
__global__ void copy_channels(const float *__restrict__ s, int ss, float *__restrict__ d, int ds,
                              int C, int64_t npix, int accumulate) {
  for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < npix * C;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t p = e / C;
    const int c = static_cast<int>(e % C);
    float v = s[p * ss + c];
    if (accumulate) v += d[p * ds + c];
    d[p * ds + c] = v;
  }
}

// MSE: loss partials and gy = 2 (y - t) / n
__global__ void mse_kernel(const float *__restrict__ y, const float *__restrict__ t,
                           float *__restrict__ gy, int64_t n, double *__restrict__ loss) {
  double s = 0.0;
  for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < n;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const float d = y[e] - t[e];
    s += static_cast<double>(d) * d;
    gy[e] = 2.f * d / static_cast<float>(n);
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(loss, s);
}

// --- BF16 mode: 8 channels (16 bytes) per thread, channel strides padded to
// 8 (lbm_net_tc.h), the padding zero; n8 = channel groups per pixel.  These
// passes run at memory speed; each does in one read and one write what a
// chain of elementwise passes would.

// (launched as a chain with the convolutions: lbm_net_tc.cu, chain_wait)
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ void unpack8(uint4 v, float (&f)[8]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int e = 0; e < 4; e++) {
    f[2 * e] = __uint_as_float(w[e] << 16);
    f[2 * e + 1] = __uint_as_float(w[e] & 0xFFFF0000u);
  }
}
__device__ __forceinline__ uint4 pack8(const float (&f)[8]) {
  uint32_t w[4];
#pragma unroll
  for (int e = 0; e < 4; e++) {
    const __nv_bfloat162 b = __floats2bfloat162_rn(f[2 * e], f[2 * e + 1]);
    w[e] = *reinterpret_cast<const uint32_t *>(&b);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ const uint4 *as8(const __nv_bfloat16 *p) {
  return reinterpret_cast<const uint4 *>(p);
}
__device__ __forceinline__ uint4 *as8(__nv_bfloat16 *p) { return reinterpret_cast<uint4 *>(p); }
// v where the ReLU output h is positive, else 0
__device__ __forceinline__ uint4 relu_gate8(uint4 v, uint4 h) {
  float f[8], g[8];
  unpack8(v, f);
  unpack8(h, g);
#pragma unroll
  for (int e = 0; e < 8; e++)
    if (!(g[e] > 0.f)) f[e] = 0.f;
  return pack8(f);
}

// d[pixel][8 n8] = s[pixel][c], zero beyond c
__global__ void __launch_bounds__(256) to_storage8(const float *__restrict__ s, int c,
                                                   __nv_bfloat16 *__restrict__ d, int n8,
                                                   int64_t npix) {
  const int64_t t = blockIdx.x * 256ll + threadIdx.x;
  if (t >= npix * n8) return;
  const int64_t p = t / n8;
  const int c0 = static_cast<int>(t - p * n8) * 8;
  float f[8];
#pragma unroll
  for (int e = 0; e < 8; e++) f[e] = c0 + e < c ? s[p * c + c0 + e] : 0.f;
  as8(d)[t] = pack8(f);
}

// 2x2 average pooling; H, W: output size
__global__ void __launch_bounds__(256) pool2_fwd8(const __nv_bfloat16 *x,
                                                  __nv_bfloat16 *y, int n8, int H,
                                                  int W, uint32_t n) {
  chain_wait();
  const uint32_t t = blockIdx.x * 256u + threadIdx.x;
  if (t >= n) return;
  const uint32_t c = t % n8, p = t / n8, j = p % W, r = p / W;  // r = image * H + row
  const uint4 *src = as8(x) + (static_cast<int64_t>(2 * r) * 2 * W + 2 * j) * n8 + c;
  const int64_t row = static_cast<int64_t>(2 * W) * n8;
  const uint4 v[4] = {src[0], src[n8], src[row], src[row + n8]};
  float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int k = 0; k < 4; k++) {
    float f[8];
    unpack8(v[k], f);
#pragma unroll
    for (int e = 0; e < 8; e++) s[e] += f[e];
  }
#pragma unroll
  for (int e = 0; e < 8; e++) s[e] *= 0.25f;
  as8(y)[t] = pack8(s);
}

// Backward of the 2x upsampling and of the ReLU below it: gx = sum of gy's
// first 8 n8 channels (stride 8 g8) over each 2x2 block, 0 where h <= 0;
// H, W: size of gx
__global__ void __launch_bounds__(256) up2_bwd8(const __nv_bfloat16 *gy, int g8,
                                                const __nv_bfloat16 *h,
                                                __nv_bfloat16 *gx, int n8, int H,
                                                int W, uint32_t n) {
  chain_wait();
  const uint32_t t = blockIdx.x * 256u + threadIdx.x;
  if (t >= n) return;
  const uint32_t c = t % n8, p = t / n8, j = p % W, r = p / W;
  const uint4 *src = as8(gy) + (static_cast<int64_t>(2 * r) * 2 * W + 2 * j) * g8 + c;
  const int64_t row = static_cast<int64_t>(2 * W) * g8;
  const uint4 v[4] = {src[0], src[g8], src[row], src[row + g8]};
  float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int k = 0; k < 4; k++) {
    float f[8];
    unpack8(v[k], f);
#pragma unroll
    for (int e = 0; e < 8; e++) s[e] += f[e];
  }
  as8(gx)[t] = relu_gate8(pack8(s), as8(h)[t]);
}

// Gradient of an encoder level's output: the skip connection's (channels
// from group g0 of gskip, stride 8 g8) plus the pooled path's (gpool / 4
// over each 2x2 block), 0 where h <= 0; H, W: size of the level
__global__ void __launch_bounds__(256) pool2_bwd8(const __nv_bfloat16 *gpool,
                                                  const __nv_bfloat16 *gskip, int g8,
                                                  int g0, const __nv_bfloat16 *h,
                                                  __nv_bfloat16 *gx, int n8, int H,
                                                  int W, uint32_t n) {
  chain_wait();
  const uint32_t t = blockIdx.x * 256u + threadIdx.x;
  if (t >= n) return;
  const uint32_t c = t % n8, p = t / n8, j = p % W, r = p / W;
  const uint4 a = as8(gpool)[(static_cast<int64_t>(r / 2) * (W / 2) + j / 2) * n8 + c];
  const uint4 b = as8(gskip)[static_cast<int64_t>(p) * g8 + g0 + c];
  float f[8], g[8];
  unpack8(a, f);
  unpack8(b, g);
#pragma unroll
  for (int e = 0; e < 8; e++) f[e] = fmaf(0.25f, f[e], g[e]);
  as8(gx)[t] = relu_gate8(pack8(f), as8(h)[t]);
}

// Squared error and its gradient gy = 2 (y - t) / n, per pixel; y, gy with
// 8 n8 channels stored, c real ones.  One atomic per CTA.
__global__ void __launch_bounds__(256) mse8(const __nv_bfloat16 *y,
                                            const float *t,
                                            __nv_bfloat16 *gy, int c, int n8,
                                            int64_t npix, double *loss) {
  chain_wait();
  double s = 0.0;
  const float n = static_cast<float>(npix * c);
  for (int64_t q = blockIdx.x * 256ll + threadIdx.x; q < npix * n8;
       q += static_cast<int64_t>(gridDim.x) * 256) {
    const int64_t p = q / n8;
    const int c0 = static_cast<int>(q - p * n8) * 8;
    float f[8];
    unpack8(as8(y)[q], f);
#pragma unroll
    for (int e = 0; e < 8; e++) {
      if (c0 + e < c) {
        const float d = f[e] - t[p * c + c0 + e];
        s += static_cast<double>(d) * d;
        f[e] = 2.f * d / n;
      } else {
        f[e] = 0.f;
      }
    }
    as8(gy)[q] = pack8(f);
  }
  __shared__ double sh[8];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; w++) s += sh[w];
    atomicAdd(loss, s);
  }
}

__global__ void adam_kernel(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, int64_t n, float lr, float b1, float b2, float eps,
                            float c1, float c2) {
  for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < n;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const float gg = g[e];
    const float mm = b1 * m[e] + (1.f - b1) * gg;
    const float vv = b2 * v[e] + (1.f - b2) * gg * gg;
    m[e] = mm;
    v[e] = vv;
    p[e] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
  }
}

int grid1(int64_t n) {
  int64_t b = (n + 255) / 256;
  return static_cast<int>(b < 1 ? 1 : (b > 65536 ? 65536 : b));
}

}  // namespace
}  // namespace net
}  // namespace lbm

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

namespace {

struct Layer {
  int ks, ci, co;
  int64_t w_off, b_off;  // offsets into the flat FP32 parameter vector
};

thread_local std::string g_net_error;

}  // namespace

struct lbm_net {
  int base = 32, levels = 4, c_in = 3, c_out = 3, precision = LBM_BF16;
  int max_batch = 1, H = 0, W = 0;
  cudaStream_t stream = nullptr;
  std::vector<Layer> layers;
  int64_t n_params = 0;
  float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
  float *wt = nullptr;  // FP32 mode: flipped weights (largest layer)
  // BF16 mode: every layer's packed weights and their adjoint's, packed from
  // the FP32 parameters when these have changed (stale); the jobs that pack
  // them (device); the weight gradient's scratch
  __nv_bfloat16 *wk = nullptr;
  std::vector<int64_t> wk_off[2];
  lbm::net::PackJob *jobs = nullptr;
  int n_jobs = 0;
  int64_t max_job = 0;
  bool stale = true;
  float *partials = nullptr;
  int sms = 1;
  // what a call reads back: the loss (a sum), and a flag that a tensor-core
  // kernel sets when one of its bounded waits runs out; device and pinned host
  struct Status {
    double loss;
    int err, pad;
  } *status = nullptr, *h_status = nullptr;
  // activations: per level encoder outputs (skip), decoder concat inputs,
  // temporaries; all storage type, sized for max_batch
  std::vector<void *> bufs;
  std::vector<int64_t> buf_elems;
  int64_t adam_t = 0;
  std::string err;
};

namespace {

size_t asize(int precision) { return precision == LBM_FP32 ? 4 : 2; }

// Buffer plan (index -> meaning), all NHWC with the channel counts below:
//   x_in                       input, c_in channels
//   e[l]a_out, e[l]b_out       encoder outputs per level (b is the skip)
//   pool[l]                    pooled input of level l (l >= 1)
//   cat[l]                     decoder input of level l: [up, skip] (BF16 mode
//                              stores only its gradient)
//   d[l]a_out, d[l]b_out
//   y                          head output
// Gradients use a second set of the same shapes.
struct Plan {
  std::vector<int64_t> elems;  // per buffer, per sample
  int x_in, y;
  std::vector<int> ea, eb, pool, cat, da, db;
};

Plan make_plan(const lbm_net_t *n) {
  Plan p;
  auto add = [&](int64_t e) {
    p.elems.push_back(e);
    return static_cast<int>(p.elems.size()) - 1;
  };
  // channels as stored (BF16 mode pads each source to a multiple of 8)
  auto st = [&](int c) { return n->precision == LBM_FP32 ? c : lbm::net::pad8(c); };
  const int64_t HW = static_cast<int64_t>(n->H) * n->W;
  p.x_in = add(HW * st(n->c_in));
  for (int l = 0; l < n->levels; l++) {
    const int64_t hw = HW >> (2 * l);
    const int ch = st(n->base << l);
    p.pool.push_back(l > 0 ? add(hw * st(n->base << (l - 1))) : -1);
    p.ea.push_back(add(hw * ch));
    p.eb.push_back(add(hw * ch));
  }
  p.cat.assign(n->levels, -1);
  p.da.assign(n->levels, -1);
  p.db.assign(n->levels, -1);
  for (int l = n->levels - 2; l >= 0; l--) {
    const int64_t hw = HW >> (2 * l);
    const int ch = st(n->base << l);
    p.cat[l] = add(hw * (st(n->base << (l + 1)) + ch));
    p.da[l] = add(hw * ch);
    p.db[l] = add(hw * ch);
  }
  p.y = add(HW * st(n->c_out));
  return p;
}

int nfail(lbm_net_t *n, int code, const std::string &m) {
  if (n) n->err = m;
  else g_net_error = m;
  return code;
}

// FP32 mode: y = act(conv(x, w) + b) with Ci inputs and Co outputs (weights
// [tap][ci][co]).
void launch_conv(lbm_net_t *n, const float *x, int xs, const float *w, const float *b, float *y,
                 int ys, int N, int H, int W, int Ci, int Co, int ks, int relu) {
  using namespace lbm::net;
  dim3 grid(((W + TP - 1) / TP) * ((H + TP - 1) / TP), (Co + TC - 1) / TC, N);
  if (ks == 3)
    conv_fwd<3><<<grid, TP * TP, 0, n->stream>>>(x, xs, w, b, y, ys, H, W, Ci, Co, relu);
  else
    conv_fwd<1><<<grid, TP * TP, 0, n->stream>>>(x, xs, w, b, y, ys, H, W, Ci, Co, relu);
}

void launch_wgrad(const lbm_net_t *n, const float *x, int xs, const float *gz, int N, int H, int W,
                  int Ci, int Co, int ks, float *dw, float *db) {
  using namespace lbm::net;
  const int64_t npix = static_cast<int64_t>(N) * H * W;
  const int chunks = static_cast<int>(std::min<int64_t>(1024, (npix + 255) / 256));
  const int per = static_cast<int>((npix + chunks - 1) / chunks);
  dim3 grid(((Ci + TC - 1) / TC) * ((Co + TC - 1) / TC), chunks);
  if (ks == 3)
    conv_bwd_weight<3><<<grid, 256, 0, n->stream>>>(x, xs, gz, N, H, W, Ci, Co, per, dw, db);
  else
    conv_bwd_weight<1><<<grid, 256, 0, n->stream>>>(x, xs, gz, N, H, W, Ci, Co, per, dw, db);
}

// FP32 mode: forward (and, if t != nullptr, loss + backward into n->grads)
cudaError_t run_fp32(lbm_net_t *n, const float *x_in, int N, const float *t, float *y_out) {
  using namespace lbm::net;
  Plan p = make_plan(n);
  const int L = n->levels;
  auto buf = [&](int i) { return static_cast<float *>(n->bufs[i]); };
  auto gbuf = [&](int i) { return static_cast<float *>(n->bufs[p.elems.size() + i]); };
  const int64_t HW = static_cast<int64_t>(n->H) * n->W;
  cudaStream_t s = n->stream;
  to_storage<<<grid1(HW * N * n->c_in), 256, 0, s>>>(x_in, buf(p.x_in), HW * N * n->c_in);
  int li = 0;
  auto W_of = [&](int k) { return n->params + n->layers[k].w_off; };
  auto B_of = [&](int k) { return n->params + n->layers[k].b_off; };
  // encoder
  const float *h = buf(p.x_in);
  int hc = n->c_in;
  for (int l = 0; l < L; l++) {
    const int H = n->H >> l, Wd = n->W >> l, ch = n->base << l;
    if (l > 0) {
      pool2_fwd<<<grid1(static_cast<int64_t>(N) * H * Wd * hc), 256, 0, s>>>(h, hc, buf(p.pool[l]), N,
                                                                             H * 2, Wd * 2, hc);
      h = buf(p.pool[l]);
    }
    launch_conv(n, h, hc, W_of(li), B_of(li), buf(p.ea[l]), ch, N, H, Wd, hc, ch, 3, 1);
    li++;
    launch_conv(n, buf(p.ea[l]), ch, W_of(li), B_of(li), buf(p.eb[l]), ch, N, H, Wd, ch, ch, 3, 1);
    li++;
    h = buf(p.eb[l]);
    hc = ch;
  }
  // decoder
  for (int l = L - 2; l >= 0; l--) {
    const int H = n->H >> l, Wd = n->W >> l, ch = n->base << l;
    const int cu = hc, ct = hc + ch;
    float *cat = buf(p.cat[l]);
    up2_fwd<<<grid1(static_cast<int64_t>(N) * H * Wd * cu), 256, 0, s>>>(h, cat, ct, N, H, Wd, cu);
    copy_channels<<<grid1(static_cast<int64_t>(N) * H * Wd * ch), 256, 0, s>>>(
        buf(p.eb[l]), ch, cat + cu, ct, ch, static_cast<int64_t>(N) * H * Wd, 0);
    launch_conv(n, cat, ct, W_of(li), B_of(li), buf(p.da[l]), ch, N, H, Wd, ct, ch, 3, 1);
    li++;
    launch_conv(n, buf(p.da[l]), ch, W_of(li), B_of(li), buf(p.db[l]), ch, N, H, Wd, ch, ch, 3, 1);
    li++;
    h = buf(p.db[l]);
    hc = ch;
  }
  const int head = li;
  launch_conv(n, h, hc, W_of(head), B_of(head), buf(p.y), n->c_out, N, n->H, n->W, hc, n->c_out, 1,
                 0);
  if (y_out)
    to_float<<<grid1(HW * N * n->c_out), 256, 0, s>>>(buf(p.y), n->c_out, y_out, n->c_out, HW * N);
  if (!t) return cudaGetLastError();

  // loss and backward
  mse_kernel<<<grid1(HW * N * n->c_out), 256, 0, s>>>(buf(p.y), t, gbuf(p.y), HW * N * n->c_out,
                                                        &n->status->loss);
  cudaMemsetAsync(n->grads, 0, n->n_params * sizeof(float), s);
  float *wt = n->wt;
  auto conv_back = [&](int k, const float *x, int xs, float *gz, float *gx, int gxs, int H, int Wd,
                       bool need_gx) {
    const Layer &ly = n->layers[k];
    launch_wgrad(n, x, xs, gz, N, H, Wd, ly.ci, ly.co, ly.ks, n->grads + ly.w_off,
                    n->grads + ly.b_off);
    if (need_gx) {
      flip_weights<<<grid1(static_cast<int64_t>(ly.ks * ly.ks) * ly.ci * ly.co), 256, 0, s>>>(
          n->params + ly.w_off, wt, ly.ks * ly.ks, ly.ci, ly.co);
      launch_conv(n, gz, ly.co, wt, nullptr, gx, gxs, N, H, Wd, ly.co, ly.ci, ly.ks, 0);
    }
  };
  // head
  {
    const Layer &ly = n->layers[head];
    (void)ly;
    conv_back(head, h, hc, gbuf(p.y), gbuf(p.db[0] >= 0 ? p.db[0] : p.eb[0]), hc, n->H, n->W, true);
  }
  // decoder backward (level 0 up to L-2)
  li = head;
  int gh_idx = p.db[0] >= 0 ? p.db[0] : p.eb[0];
  for (int l = 0; l <= L - 2; l++) {
    const int H = n->H >> l, Wd = n->W >> l, ch = n->base << l;
    const int cu = ch * 2, ct = cu + ch;
    const int kb = head - 1 - 2 * l, ka = kb - 1;
    // through d_l b
    relu_mask<<<grid1(static_cast<int64_t>(N) * H * Wd * ch), 256, 0, s>>>(
        gbuf(gh_idx), buf(p.db[l]), static_cast<int64_t>(N) * H * Wd * ch);
    conv_back(kb, buf(p.da[l]), ch, gbuf(gh_idx), gbuf(p.da[l]), ch, H, Wd, true);
    relu_mask<<<grid1(static_cast<int64_t>(N) * H * Wd * ch), 256, 0, s>>>(
        gbuf(p.da[l]), buf(p.da[l]), static_cast<int64_t>(N) * H * Wd * ch);
    conv_back(ka, buf(p.cat[l]), ct, gbuf(p.da[l]), gbuf(p.cat[l]), ct, H, Wd, true);
    // split the concat gradient: skip part into the encoder level-l output grad,
    // upsampled part into the grad of the level-(l+1) output
    copy_channels<<<grid1(static_cast<int64_t>(N) * H * Wd * ch), 256, 0, s>>>(
        gbuf(p.cat[l]) + cu, ct, gbuf(p.eb[l]), ch, ch, static_cast<int64_t>(N) * H * Wd, 0);
    const int up_idx = (l + 1 <= L - 2) ? p.db[l + 1] : p.eb[L - 1];
    up2_bwd<<<grid1(static_cast<int64_t>(N) * (H / 2) * (Wd / 2) * cu), 256, 0, s>>>(
        gbuf(p.cat[l]), ct, gbuf(up_idx), N, H, Wd, cu);
    gh_idx = up_idx;
  }
  // encoder backward (level L-1 down to 0); gbuf(eb[l]) for l < L-1 already
  // holds the skip gradient, to which the pooled-path gradient is added
  for (int l = L - 1; l >= 0; l--) {
    const int H = n->H >> l, Wd = n->W >> l, ch = n->base << l;
    const int ka = 2 * l, kb = 2 * l + 1;
    const int cin = l == 0 ? n->c_in : (n->base << (l - 1));
    relu_mask<<<grid1(static_cast<int64_t>(N) * H * Wd * ch), 256, 0, s>>>(
        gbuf(p.eb[l]), buf(p.eb[l]), static_cast<int64_t>(N) * H * Wd * ch);
    conv_back(kb, buf(p.ea[l]), ch, gbuf(p.eb[l]), gbuf(p.ea[l]), ch, H, Wd, true);
    relu_mask<<<grid1(static_cast<int64_t>(N) * H * Wd * ch), 256, 0, s>>>(
        gbuf(p.ea[l]), buf(p.ea[l]), static_cast<int64_t>(N) * H * Wd * ch);
    const float *xin = l == 0 ? buf(p.x_in) : buf(p.pool[l]);
    conv_back(ka, xin, cin, gbuf(p.ea[l]), l == 0 ? nullptr : gbuf(p.pool[l]), cin, H, Wd, l > 0);
    if (l > 0)
      pool2_bwd<<<grid1(static_cast<int64_t>(N) * H * 2 * Wd * 2 * cin), 256, 0, s>>>(
          gbuf(p.pool[l]), gbuf(p.eb[l - 1]), cin, N, H * 2, Wd * 2, cin, 1);
  }
  return cudaGetLastError();
}

// BF16 mode: the same on the tensor cores (lbm_net_tc.cu).  Activations have
// padded channel strides; the decoder's concatenated input is read from its
// two sources, and every stored gradient is already masked by its ReLU.
cudaError_t run_bf16(lbm_net_t *n, const float *x_in, int N, const float *t, float *y_out) {
  using namespace lbm::net;
  using B16 = __nv_bfloat16;
  const Plan p = make_plan(n);
  const int L = n->levels;
  const int64_t HW = static_cast<int64_t>(n->H) * n->W;
  cudaStream_t s = n->stream;
  cudaError_t e = cudaSuccess;
  auto buf = [&](int i) { return static_cast<B16 *>(n->bufs[i]); };
  auto gbuf = [&](int i) { return static_cast<B16 *>(n->bufs[p.elems.size() + i]); };
  auto blocks = [](int64_t k) { return static_cast<unsigned>((k + 255) / 256); };
  if (n->stale) {
    e = launch_pack(n->jobs, n->n_jobs, n->max_job, s);
    if (e != cudaSuccess) return e;
    n->stale = false;
  }
  auto conv = [&](int k, ConvInput in, int H, int W, int relu, B16 *y, float *yf) {
    if (e != cudaSuccess) return;
    const Layer &ly = n->layers[k];
    ConvCall c;
    c.in = in;
    c.ks = ly.ks;
    c.N = N;
    c.H = H;
    c.W = W;
    c.co = ly.co;
    c.wk = n->wk + n->wk_off[0][k];
    c.bias = n->params + ly.b_off;
    c.relu = relu;
    c.y = y;
    c.yf = yf;
    e = launch_conv_tc(c, n->sms, &n->status->err, s);
  };
  auto single = [](const B16 *x, int c) {
    ConvInput in;
    in.xa = x;
    in.ca = c;
    return in;
  };
  const int n8x = pad8(n->c_in) / 8;
  to_storage8<<<blocks(HW * N * n8x), 256, 0, s>>>(x_in, n->c_in, buf(p.x_in), n8x, HW * N);
  // encoder
  for (int l = 0; l < L; l++) {
    const int H = n->H >> l, W = n->W >> l, ch = n->base << l;
    ConvInput in = single(buf(p.x_in), n->c_in);
    if (l > 0) {
      const int cb = n->base << (l - 1), n8 = pad8(cb) / 8;
      const int64_t k = static_cast<int64_t>(N) * H * W * n8;
      if (e == cudaSuccess)
        e = lbm::launch_chained(pool2_fwd8, dim3(blocks(k)), 256, 0, s, buf(p.eb[l - 1]),
                                buf(p.pool[l]), n8, H, W, static_cast<uint32_t>(k));
      in = single(buf(p.pool[l]), cb);
    }
    conv(2 * l, in, H, W, 1, buf(p.ea[l]), nullptr);
    conv(2 * l + 1, single(buf(p.ea[l]), ch), H, W, 1, buf(p.eb[l]), nullptr);
  }
  // the decoder's input at level l: the level below upsampled, then the skip
  auto below = [&](int l) { return l + 1 <= L - 2 ? p.db[l + 1] : p.eb[L - 1]; };
  auto cat_in = [&](int l) {
    ConvInput in = single(buf(below(l)), n->base << (l + 1));
    in.up = 1;
    in.xb = buf(p.eb[l]);
    in.cb = n->base << l;
    return in;
  };
  int li = 2 * L;
  for (int l = L - 2; l >= 0; l--) {
    const int H = n->H >> l, W = n->W >> l, ch = n->base << l;
    conv(li++, cat_in(l), H, W, 1, buf(p.da[l]), nullptr);
    conv(li++, single(buf(p.da[l]), ch), H, W, 1, buf(p.db[l]), nullptr);
  }
  const int head = li;
  const int top = L > 1 ? p.db[0] : p.eb[0];
  conv(head, single(buf(top), n->base), n->H, n->W, 0, buf(p.y), y_out);
  if (e != cudaSuccess || !t) return e != cudaSuccess ? e : cudaGetLastError();

  // loss and backward
  const int n8y = pad8(n->c_out) / 8;
  e = lbm::launch_chained(mse8, dim3(std::min<unsigned>(blocks(HW * N * n8y), 4u * n->sms)), 256, 0,
                          s, buf(p.y), t, gbuf(p.y), n->c_out, n8y, HW * N, &n->status->loss);
  // gradients of layer k from its input and its (masked) output gradient gz;
  // gx: the input's gradient, 0 where mask <= 0 (may be null)
  auto back = [&](int k, const ConvInput &in, const B16 *gz, B16 *gx, const B16 *mask, int H,
                  int W) {
    if (e != cudaSuccess) return;
    const Layer &ly = n->layers[k];
    e = launch_wgrad_tc(in, ly.ks, gz, ly.co, N, H, W, n->partials, n->grads + ly.w_off, n->sms,
                        &n->status->err, s);
    if (e != cudaSuccess || !gx) return;
    ConvCall c;
    c.in = single(gz, ly.co);
    c.ks = ly.ks;
    c.N = N;
    c.H = H;
    c.W = W;
    c.co = in.padded();
    c.wk = n->wk + n->wk_off[1][k];
    c.mask = mask;
    c.y = gx;
    e = launch_conv_tc(c, n->sms, &n->status->err, s);
  };
  back(head, single(buf(top), n->base), gbuf(p.y), gbuf(top), buf(top), n->H, n->W);
  for (int l = 0; l <= L - 2; l++) {
    const int H = n->H >> l, W = n->W >> l, ch = n->base << l;
    const int kb = head - 1 - 2 * l, ka = kb - 1;
    back(kb, single(buf(p.da[l]), ch), gbuf(p.db[l]), gbuf(p.da[l]), buf(p.da[l]), H, W);
    const ConvInput in = cat_in(l);
    back(ka, in, gbuf(p.da[l]), gbuf(p.cat[l]), nullptr, H, W);
    const int n8 = pad8(in.ca) / 8;
    const int64_t k = static_cast<int64_t>(N) * (H / 2) * (W / 2) * n8;
    if (e == cudaSuccess)
      e = lbm::launch_chained(up2_bwd8, dim3(blocks(k)), 256, 0, s, gbuf(p.cat[l]),
                              in.padded() / 8, buf(below(l)), gbuf(below(l)), n8, H / 2, W / 2,
                              static_cast<uint32_t>(k));
  }
  for (int l = L - 1; l >= 0; l--) {
    const int H = n->H >> l, W = n->W >> l, ch = n->base << l;
    if (l < L - 1) {  // the deepest level's gradient came from up2_bwd8
      const ConvInput in = cat_in(l);
      const int n8 = pad8(ch) / 8;
      const int64_t k = static_cast<int64_t>(N) * H * W * n8;
      if (e == cudaSuccess)
        e = lbm::launch_chained(pool2_bwd8, dim3(blocks(k)), 256, 0, s, gbuf(p.pool[l + 1]),
                                gbuf(p.cat[l]), in.padded() / 8, pad8(in.ca) / 8, buf(p.eb[l]),
                                gbuf(p.eb[l]), n8, H, W, static_cast<uint32_t>(k));
    }
    back(2 * l + 1, single(buf(p.ea[l]), ch), gbuf(p.eb[l]), gbuf(p.ea[l]), buf(p.ea[l]), H, W);
    if (l > 0)
      back(2 * l, single(buf(p.pool[l]), n->base << (l - 1)), gbuf(p.ea[l]), gbuf(p.pool[l]),
           nullptr, H, W);
    else
      back(0, single(buf(p.x_in), n->c_in), gbuf(p.ea[0]), nullptr, nullptr, H, W);
  }
  return e != cudaSuccess ? e : cudaGetLastError();
}

// One pass and its status (loss, bounded waits) read back; synchronises.
int run(lbm_net_t *n, const float *x, int N, const float *t, float *y, double *loss) {
  cudaError_t e = cudaMemsetAsync(n->status, 0, sizeof(*n->status), n->stream);
  if (e == cudaSuccess)
    e = n->precision == LBM_FP32 ? run_fp32(n, x, N, t, y) : run_bf16(n, x, N, t, y);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(n->h_status, n->status, sizeof(*n->status), cudaMemcpyDeviceToHost,
                        n->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(n->stream);
  if (e != cudaSuccess) return nfail(n, LBM_ECUDA, cudaGetErrorString(e));
  if (n->h_status->err)
    return nfail(n, LBM_ETIMEOUT, "a tensor-core convolution's bounded wait ran out");
  if (loss)
    *loss = n->h_status->loss /
            static_cast<double>(static_cast<int64_t>(n->H) * n->W * N * n->c_out);
  return LBM_OK;
}

}  // namespace

extern "C" {

int lbm_net_create(int32_t base, int32_t levels, int32_t c_in, int32_t c_out, int32_t precision,
                   int32_t max_batch, int32_t H, int32_t W, uint64_t seed, void *stream,
                   lbm_net_t **out) {
  g_net_error.clear();
  if (!out) return nfail(nullptr, LBM_EINVAL, "null argument");
  *out = nullptr;
  if (base < 1 || levels < 1 || levels > 8 || c_in < 1 || c_out < 1 || max_batch < 1 || H < 1 ||
      W < 1)
    return nfail(nullptr, LBM_EINVAL, "bad network shape");
  if (precision != LBM_FP32 && precision != LBM_BF16)
    return nfail(nullptr, LBM_EINVAL, "network precision must be LBM_FP32 or LBM_BF16");
  if ((H % (1 << (levels - 1))) || (W % (1 << (levels - 1))))
    return nfail(nullptr, LBM_EINVAL, "H and W must be divisible by 2^(levels-1)");
  lbm_net_t *n = new (std::nothrow) lbm_net_t();
  if (!n) return nfail(nullptr, LBM_ENOMEM, "host allocation failed");
  n->base = base;
  n->levels = levels;
  n->c_in = c_in;
  n->c_out = c_out;
  n->precision = precision;
  n->max_batch = max_batch;
  n->H = H;
  n->W = W;
  n->stream = static_cast<cudaStream_t>(stream);
  // layers in parameter order (the order of the FP64 reference)
  int64_t off = 0;
  int prev = c_in;
  int64_t max_w = 0;
  auto add = [&](int ks, int ci, int co) {
    Layer ly{ks, ci, co, off, off + static_cast<int64_t>(ks) * ks * ci * co};
    off = ly.b_off + co;
    max_w = std::max<int64_t>(max_w, static_cast<int64_t>(ks) * ks * ci * co);
    n->layers.push_back(ly);
  };
  for (int l = 0; l < levels; l++) {
    add(3, prev, base << l);
    add(3, base << l, base << l);
    prev = base << l;
  }
  for (int l = levels - 2; l >= 0; l--) {
    add(3, (base << (l + 1)) + (base << l), base << l);
    add(3, base << l, base << l);
  }
  add(1, base, c_out);
  n->n_params = off;
  Plan p = make_plan(n);
  const size_t as = asize(precision);
  cudaError_t e = cudaSuccess;
  for (float **ptr : {&n->params, &n->grads, &n->m, &n->v})
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void **>(ptr), off * sizeof(float));
  int dev = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n->sms, cudaDevAttrMultiProcessorCount, dev);
  if (precision == LBM_FP32) {
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void **>(&n->wt), max_w * sizeof(float));
  } else {
    // packed weights of every layer and of its adjoint (the first layer's
    // adjoint is never needed), and the largest weight-gradient scratch
    std::vector<lbm::net::PackJob> jobs;
    int64_t wk = 0, scratch = 1;
    for (size_t k = 0; k < n->layers.size(); k++) {
      const Layer &ly = n->layers[k];
      const int dec = static_cast<int>(k) - 2 * levels;  // >= 0: decoder layers, then the head
      const bool cat = k + 1 < n->layers.size() && dec >= 0 && dec % 2 == 0;
      const int cb = cat ? ly.co : 0, ca = ly.ci - cb;
      const int padded = lbm::net::pad8(ca) + lbm::net::pad8(cb);
      const int lev = dec < 0 ? static_cast<int>(k) / 2
                              : std::max(0, levels - 2 - dec / 2);  // the head: level 0
      scratch = std::max(scratch, lbm::net::wgrad_scratch(ly.ks, ly.ci, padded, ly.co, max_batch,
                                                          H >> lev, W >> lev, n->sms));
      for (int flip = 0; flip < 2; flip++) {
        const int64_t el = flip ? lbm::net::packed_elems(ly.ks, lbm::net::pad8(ly.co), padded)
                                : lbm::net::packed_elems(ly.ks, padded, ly.co);
        n->wk_off[flip].push_back(wk);
        if (flip && k == 0) continue;
        jobs.push_back({n->params + ly.w_off, reinterpret_cast<__nv_bfloat16 *>(wk), ly.ks, ca, cb,
                        ly.co, flip, el});
        n->max_job = std::max(n->max_job, el);
        wk += (el + 63) / 64 * 64;
      }
    }
    n->n_jobs = static_cast<int>(jobs.size());
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void **>(&n->wk), wk * 2);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void **>(&n->partials), scratch * 4);
    for (auto &j : jobs) j.out = n->wk + reinterpret_cast<intptr_t>(j.out);
    if (e == cudaSuccess)
      e = cudaMalloc(reinterpret_cast<void **>(&n->jobs), jobs.size() * sizeof(jobs[0]));
    if (e == cudaSuccess)
      e = cudaMemcpy(n->jobs, jobs.data(), jobs.size() * sizeof(jobs[0]), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = lbm::net::setup_tc();
  }
  if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void **>(&n->status), sizeof(*n->status));
  if (e == cudaSuccess)
    e = cudaMallocHost(reinterpret_cast<void **>(&n->h_status), sizeof(*n->h_status));
  for (int g = 0; g < 2 && e == cudaSuccess; g++)
    for (size_t i = 0; i < p.elems.size() && e == cudaSuccess; i++) {
      void *b = nullptr;
      // (BF16 mode reads the decoder's inputs from their sources)
      const bool cat = std::find(p.cat.begin(), p.cat.end(), static_cast<int>(i)) != p.cat.end();
      if (g == 1 || !cat || precision == LBM_FP32) e = cudaMalloc(&b, p.elems[i] * max_batch * as);
      n->bufs.push_back(b);
    }
  if (e == cudaSuccess) e = cudaMemset(n->m, 0, off * sizeof(float));
  if (e == cudaSuccess) e = cudaMemset(n->v, 0, off * sizeof(float));
  if (e == cudaSuccess) {
    // He-normal weights from a counter-based generator (splitmix64 + Box-Muller), zero biases
    std::vector<float> hp(off, 0.f);
    uint64_t st = seed * 0x9E3779B97F4A7C15ull + 1;
    auto next = [&]() {
      uint64_t z = (st += 0x9E3779B97F4A7C15ull);
      z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
      z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
      z ^= z >> 31;
      return (static_cast<double>(z >> 11) + 0.5) * (1.0 / 9007199254740992.0);
    };
    for (const Layer &ly : n->layers) {
      const double sd = std::sqrt(2.0 / (ly.ks * ly.ks * ly.ci));
      for (int64_t q = ly.w_off; q < ly.b_off; q++) {
        const double u1 = next(), u2 = next();
        hp[q] = static_cast<float>(sd * std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2));
      }
    }
    e = cudaMemcpy(n->params, hp.data(), off * sizeof(float), cudaMemcpyHostToDevice);
  }
  if (e != cudaSuccess) {
    g_net_error = std::string("device setup: ") + cudaGetErrorString(e);
    lbm_net_destroy(n);
    return LBM_ECUDA;
  }
  *out = n;
  return LBM_OK;
}

int64_t lbm_net_num_params(const lbm_net_t *n) { return n ? n->n_params : -1; }

int lbm_net_set_params(lbm_net_t *n, const float *params, int64_t count) {
  if (!n || !params || count != n->n_params) return nfail(n, LBM_EINVAL, "parameter count mismatch");
  cudaError_t e = cudaMemcpy(n->params, params, count * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(n->m, 0, count * sizeof(float));
  if (e == cudaSuccess) e = cudaMemset(n->v, 0, count * sizeof(float));
  n->stale = true;
  n->adam_t = 0;
  return e == cudaSuccess ? LBM_OK : nfail(n, LBM_ECUDA, cudaGetErrorString(e));
}

int lbm_net_get_params(const lbm_net_t *n, float *params, int64_t count) {
  if (!n || !params || count != n->n_params) return LBM_EINVAL;
  return cudaMemcpy(params, n->params, count * sizeof(float), cudaMemcpyDeviceToHost) == cudaSuccess
             ? LBM_OK
             : LBM_ECUDA;
}

int lbm_net_forward(lbm_net_t *n, const float *x, int32_t batch, float *y) {
  if (!n || !x || !y || batch < 1 || batch > n->max_batch) return nfail(n, LBM_EINVAL, "bad batch");
  return run(n, x, batch, nullptr, y, nullptr);
}

int lbm_net_gradients(lbm_net_t *n, const float *x, const float *t, int32_t batch, float *grads,
                      double *loss) {
  if (!n || !x || !t || batch < 1 || batch > n->max_batch) return nfail(n, LBM_EINVAL, "bad batch");
  double l = 0.0;
  const int rc = run(n, x, batch, t, nullptr, &l);
  if (rc != LBM_OK) return rc;
  if (loss) *loss = l;
  if (!grads) return LBM_OK;
  const cudaError_t e =
      cudaMemcpy(grads, n->grads, n->n_params * sizeof(float), cudaMemcpyDeviceToHost);
  return e == cudaSuccess ? LBM_OK : nfail(n, LBM_ECUDA, cudaGetErrorString(e));
}

int lbm_net_train_step(lbm_net_t *n, const float *x, const float *t, int32_t batch, float lr,
                       double *loss) {
  int rc = lbm_net_gradients(n, x, t, batch, nullptr, loss);
  if (rc) return rc;
  n->adam_t++;
  n->stale = true;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, static_cast<float>(n->adam_t));
  const float c2 = 1.f - std::pow(b2, static_cast<float>(n->adam_t));
  lbm::net::adam_kernel<<<lbm::net::grid1(n->n_params), 256, 0, n->stream>>>(
      n->params, n->grads, n->m, n->v, n->n_params, lr, b1, b2, 1e-8f, c1, c2);
  cudaError_t e = cudaStreamSynchronize(n->stream);
  return e == cudaSuccess ? LBM_OK : nfail(n, LBM_ECUDA, cudaGetErrorString(e));
}

void lbm_net_destroy(lbm_net_t *n) {
  if (!n) return;
  cudaStreamSynchronize(n->stream);
  for (void *p : {static_cast<void *>(n->params), static_cast<void *>(n->grads),
                  static_cast<void *>(n->m), static_cast<void *>(n->v), static_cast<void *>(n->wt),
                  static_cast<void *>(n->wk), static_cast<void *>(n->jobs),
                  static_cast<void *>(n->partials), static_cast<void *>(n->status)})
    if (p) cudaFree(p);
  if (n->h_status) cudaFreeHost(n->h_status);
  for (void *b : n->bufs)
    if (b) cudaFree(b);
  delete n;
}

const char *lbm_net_last_error(const lbm_net_t *n) { return n ? n->err.c_str() : g_net_error.c_str(); }

}  // extern "C"
