// Tensor-core kernels of the warm-start network's BF16 mode (lbm_net_tc.cu)
// as the network's host side (lbm_net.cu) calls them.
//
// Every BF16 activation is NHWC with its channel count padded to a multiple
// of 8 (pad8); the padding channels hold zeros.
#pragma once

#include <cstdint>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace lbm {
namespace net {

#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int pad8(int c) { return (c + 7) / 8 * 8; }
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int pad16(int c) { return (c + 15) / 16 * 16; }

// The input of a convolution: channels [0, ca) of xa, then those of xb (a
// concatenation that is never stored).  xa may be a tensor of half the
// height and width, upsampled by repetition (up = 1).
struct ConvInput {
  const __nv_bfloat16 *xa = nullptr;
  int ca = 0;   // channels of xa; its pixel stride is pad8(ca)
  int up = 0;
  const __nv_bfloat16 *xb = nullptr;
  int cb = 0;   // channels of xb (0: none)
  int padded() const { return pad8(ca) + pad8(cb); }  // channels as the kernels see them
};

// y = act(conv(x, w) + b), ks x ks taps, zero padding outside the image.
struct ConvCall {
  ConvInput in;
  int ks = 3, N = 0, H = 0, W = 0;
  int co = 0;                     // channels of y as stored: pixel stride pad8(co)
  const __nv_bfloat16 *wk = nullptr;  // packed weights (pack_all)
  const float *bias = nullptr;    // per output channel (plain order), or null
  int relu = 0;
  const __nv_bfloat16 *mask = nullptr;  // same shape as y: y = 0 where mask <= 0; or null
  __nv_bfloat16 *y = nullptr;
  float *yf = nullptr;            // also y in FP32, pixel stride co; or null
};

// Output-channel tile (a multiple of 16, at most 128) of a convolution with
// `co` outputs: as few tiles as possible, of even size (192 -> 2 x 96).
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int conv_tile_n(int co) {
  return pad16((pad16(co) + (pad16(co) + 127) / 128 - 1) / ((pad16(co) + 127) / 128));
}
// Elements of the packed weights of a convolution with `ci` (padded) inputs
// and `co` outputs.
int64_t packed_elems(int ks, int ci_padded, int co);

// One convolution's weights to pack from the FP32 parameters: the layer
// itself (flip = 0) or its adjoint (flip = 1: taps reversed, inputs and
// outputs exchanged).  ca, cb: the layer's input channels per source.
struct PackJob {
  const float *w;
  __nv_bfloat16 *out;
  int ks, ca, cb, co, flip;
  int64_t elems;
};
cudaError_t launch_pack(const PackJob *jobs_dev, int n_jobs, int64_t max_elems, cudaStream_t s);

cudaError_t setup_tc();  // kernel attributes, once per device
cudaError_t launch_conv_tc(const ConvCall &c, int sms, int *err, cudaStream_t s);

// Weight and bias gradients: dw[(tap, ci, co)] then db[co], from the layer's
// input and its masked output gradient gz (pixel stride pad8(co)).
// partials: scratch of wgrad_scratch floats.
int64_t wgrad_scratch(int ks, int ci, int ci_padded, int co, int N, int H, int W, int sms);
cudaError_t launch_wgrad_tc(const ConvInput &in, int ks, const __nv_bfloat16 *gz, int co, int N,
                            int H, int W, float *partials, float *dw, int sms, int *err,
                            cudaStream_t s);

}  // namespace net
}  // namespace lbm
