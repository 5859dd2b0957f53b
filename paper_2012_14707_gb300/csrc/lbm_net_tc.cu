// Convolutions of the warm-start network's BF16 mode on the tcgen05 tensor
// cores: forward and backward-data (conv_halo_tc) and the weight gradient
// (wgrad_tc), with the packing of their weights.
//
// Shared-memory layout of an image tile (both kernels): the tile's pixels
// with the halo its taps reach, as "slabs" of 8 channels -- slab c8 holds
// 16 bytes (8 BF16 channels) per pixel, pixels row by row.  In the tensor
// cores' canonical layout without swizzle a core matrix is 8 rows of 16
// contiguous bytes, rows 16 bytes apart: 8 neighbouring pixels of a slab are
// one core matrix, whatever pixel it starts at.  So a tap's shifted operand
// is the same tile with another start address, and each input element is
// copied to shared memory once per tile instead of once per tap.  Read with
// the channels as K (K-major) the tile is the forward operand, with the
// pixels as K (MN-major) it is the weight gradient's.  A slab's length is an
// odd number of 16-byte units, so the copies of a pixel's slabs fall in
// different banks.
//
// Every wait is bounded; one that runs out sets *err, and the CTA's roles
// give up in turn after waiting for the copies they started.
#include <algorithm>
#include <cstdint>

#include "lbm_net_tc.h"

namespace lbm {
namespace net {
namespace {

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(count)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}
constexpr int kWaitLimit = 1 << 24;  // polls: a fraction of a second
// Waits for the phase with parity `phase`; false if it did not come within
// kWaitLimit polls (test_wait: each poll returns at once) or the CTA gave up.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t phase, volatile int *gave_up) {
  const uint32_t a = smem_addr(bar);
  for (int it = 0; it < kWaitLimit; it++) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(a), "r"(phase)
        : "memory");
    if (done) return true;
    if ((it & 1023) == 1023 && *gave_up) return false;
  }
  return false;
}

// Shared-memory matrix descriptor without swizzle; lbo, sbo in bytes.
// K-major operand: lbo between core matrices along K, sbo between groups of
// 8 rows.  MN-major operand: sbo between core matrices along M (N), lbo
// between groups of 8 along K.  Bit 46: descriptor version.
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return static_cast<uint64_t>((addr >> 4) & 0x3FFFu) |
         (static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16) |
         (static_cast<uint64_t>((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}
// kind::f16, D = FP32, A = B = BF16, M = 128; mn: both operands MN-major
__host__ __device__ constexpr uint32_t umma_idesc(int N, bool mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (mn ? (1u << 15) | (1u << 16) : 0u) |
         (static_cast<uint32_t>(N >> 3) << 17) | (static_cast<uint32_t>(128 >> 4) << 24);
}
__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                         bool accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate ? 1u : 0u)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                   smem_addr(bar))
               : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                   smem_addr(slot)),
               "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t addr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(addr), "r"(cols)
               : "memory");
}
__device__ __forceinline__ void fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
}
// 16 columns of this warp's 32 lanes of D
__device__ __forceinline__ void tmem_ld16(uint32_t addr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(addr));
}
__device__ __forceinline__ void tmem_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src),
               "r"(valid ? 16u : 0u)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
__device__ __forceinline__ void fence_async_proxy() {
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes,
                                          uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
          dst),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// Both sources of a convolution's input, in slabs.
struct InputDev {
  const __nv_bfloat16 *xa, *xb;
  int sa, sb;        // pixel strides (elements)
  int n8a, n8;       // slabs of xa, of both
  int up;
};
// The 8 channels of slab c8 of pixel (n, i, j) of an H x W image.
__device__ __forceinline__ const __nv_bfloat16 *input_at(const InputDev &x, int n, int i, int j,
                                                         int H, int W, int c8) {
  if (c8 < x.n8a) {
    const int Ha = H >> x.up, Wa = W >> x.up;
    return x.xa + (static_cast<int64_t>((n * Ha + (i >> x.up)) * Wa + (j >> x.up)) * x.sa + c8 * 8);
  }
  return x.xb + (static_cast<int64_t>((n * H + i) * W + j) * x.sb + (c8 - x.n8a) * 8);
}

// ---------------------------------------------------------------------------
// Forward and backward-data convolution
// ---------------------------------------------------------------------------
// D[p][o] = sum over taps d, channels c of X[p + d][c] W[o][d][c], taps
// outermost, channels in order (every tile shape below sums in this order, so
// they all give the same bits; an input of more channels than shared memory
// takes of a tile, about 500, is copied part by part for every tap).  A CTA keeps one block of NT output channels
// and walks over image tiles of MT x (8 x 16) pixels.  Roles: one lane copies
// packed weights (bulk copies; all of them once where they fit beside the
// image tiles, else through a ring, tap by tap in chunks of 64 channels),
// four warps copy image tiles (cp.async, zero outside the image), one lane
// issues the MMAs (M = 128 pixels, N = NT, K = 16), four warps read the
// accumulators back, of which there are two sets, so that a tile's epilogue
// overlaps the next tile's MMAs.
constexpr int kConvThreads = 320;
constexpr int kMaxStagesB = 54;   // 9 taps x 6 chunks of 64: every weight block resident
constexpr int kMaxStagesA = 3;
constexpr int kSmemMax = 232448 - 2048;  // dynamic shared memory a CTA may use (static below)

struct ConvDev {
  InputDev x;
  int k8;                 // slabs the MMAs run over (even; those >= x.n8 are zero)
  // ... in `parts` parts of p8 slabs, as many as shared memory takes at once;
  // one part: a tile is copied once for all taps; more: again for every tap
  int parts, p8, unit_taps;
  uint32_t magic, magic_last;  // 2^32 / slabs + 1 of a part and of the last one
  const __nv_bfloat16 *wk;
  const float *bias;
  const __nv_bfloat16 *mask;
  __nv_bfloat16 *y;
  float *yf;
  int N, H, W, co, cos;   // output channels and their stored stride
  int NT, relu;
  int tiles_x, tiles_y, tiles;
  int stages_a, stages_b, resident;
  uint32_t tmem_cols;
  int *err;
};

template <int KS, int MT>
struct TileShape {
  static constexpr int kHalo = KS / 2;
  static constexpr int kW = 8 * MT, kH = 16;
  static constexpr int kWp = kW + 2 * kHalo, kHp = kH + 2 * kHalo;
  static constexpr int kPix = kWp * kHp;
  static constexpr uint32_t kSlab = (kPix | 1) * 16;
};

template <int KS, int MT>
__global__ void __launch_bounds__(kConvThreads, 1) conv_halo_tc(const __grid_constant__ ConvDev a) {
  using S = TileShape<KS, MT>;
  extern __shared__ __align__(128) unsigned char dyn[];
  __shared__ uint64_t full_a[kMaxStagesA], empty_a[kMaxStagesA];
  __shared__ uint64_t full_b[kMaxStagesB], empty_b[kMaxStagesB];
  __shared__ uint64_t full_d[2], empty_d[2], drained;
  __shared__ uint32_t tmem_slot;
  __shared__ int gave_up;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t a_bytes = static_cast<uint32_t>(a.p8) * S::kSlab;
  const uint32_t b_bytes = static_cast<uint32_t>(a.NT) * 128u;  // 64 channels
  const uint32_t base_a = smem_addr(dyn);
  const uint32_t base_b = base_a + static_cast<uint32_t>(a.stages_a) * ((a_bytes + 127u) & ~127u);
  const uint32_t stride_a = (a_bytes + 127u) & ~127u;
  if (threadIdx.x == 0) {
    for (int i = 0; i < a.stages_a; i++) {
      mbar_init(&full_a[i], 128);
      mbar_init(&empty_a[i], 1);
    }
    for (int i = 0; i < a.stages_b; i++) {
      mbar_init(&full_b[i], 1);
      mbar_init(&empty_b[i], 1);
    }
    for (int i = 0; i < 2; i++) {
      mbar_init(&full_d[i], 1);
      mbar_init(&empty_d[i], 128);
    }
    mbar_init(&drained, 1);
    gave_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 1) tmem_alloc(&tmem_slot, a.tmem_cols);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_slot;

  if (warp == 0) {
    // weights
    if (lane == 0) {
      const unsigned char *src = reinterpret_cast<const unsigned char *>(a.wk) +
                                 static_cast<int64_t>(blockIdx.y) * KS * KS * a.k8 * a.NT * 16;
      int st = 0, issued = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < a.tiles; t += gridDim.x) {
        const int units = a.parts * (KS * KS / a.unit_taps);
        for (int u = 0; ok && u < units; u++) {
          const int t0 = u / a.parts * a.unit_taps, p = u % a.parts;
          const int k8 = min(a.p8, a.k8 - p * a.p8), chunks = (k8 + 7) / 8;
          for (int b = 0; b < a.unit_taps * chunks; b++) {
            if (issued >= a.stages_b && !mbar_wait(&empty_b[st], ph ^ 1u, &gave_up)) {
              ok = false;
              break;
            }
            const int tap = t0 + b / chunks, c8 = (b % chunks) * 8;
            const uint32_t bytes = static_cast<uint32_t>(min(8, k8 - c8)) * a.NT * 16u;
            mbar_expect(&full_b[st], bytes);
            bulk_copy(base_b + st * b_bytes,
                      src + static_cast<int64_t>(tap * a.k8 + p * a.p8 + c8) * a.NT * 16, bytes,
                      &full_b[st]);
            issued++;
            if (++st == a.stages_b) {
              st = 0;
              ph ^= 1u;
            }
          }
        }
        if (a.resident) break;
      }
      if (!ok) {
        gave_up = 1;
        atomicExch(a.err, 1);
        // the copies in flight land before the CTA ends
        int never = 0;
        for (int i = max(0, issued - a.stages_b); i < issued; i++)
          mbar_wait(&full_b[i % a.stages_b], (i / a.stages_b) & 1, &never);
      }
    }
  } else if (warp == 1) {
    // MMAs
    if (lane == 0) {
      const uint32_t idesc = umma_idesc(a.NT, false);
      const uint32_t lbo_b = static_cast<uint32_t>(a.NT) * 16u;
      int sa = 0, sb = 0, it = 0;
      uint32_t pa = 0, pb = 0;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < a.tiles; t += gridDim.x, it++) {
        const int acc = it & 1;
        if (it >= 2 && !mbar_wait(&empty_d[acc], ((it >> 1) & 1) ^ 1u, &gave_up)) {
          ok = false;
          break;
        }
        const uint32_t d0 = tmem + static_cast<uint32_t>(acc * MT * a.NT);
        if (a.resident) {
          sb = 0;
          pb = 0;
        }
        bool first = true;
        const int units = a.parts * (KS * KS / a.unit_taps);
        for (int u = 0; ok && u < units; u++) {
          if (!mbar_wait(&full_a[sa], pa, &gave_up)) {
            ok = false;
            break;
          }
          fence_after();
          const uint32_t ta = base_a + sa * stride_a;
          const int t0 = u / a.parts * a.unit_taps, p = u % a.parts;
          const int k8 = min(a.p8, a.k8 - p * a.p8), chunks = (k8 + 7) / 8;
          for (int tap = t0; ok && tap < t0 + a.unit_taps; tap++) {
            const uint32_t shift = static_cast<uint32_t>((tap / KS) * S::kWp + (tap % KS)) * 16u;
            for (int ch = 0; ch < chunks; ch++) {
              if (!mbar_wait(&full_b[sb], pb, &gave_up)) {
                ok = false;
                break;
              }
              fence_after();
              const int k16 = min(8, k8 - ch * 8) / 2;
              const uint32_t tb = base_b + sb * b_bytes;
              for (int k = 0; k < k16; k++) {
                const uint64_t bd = umma_desc(tb + k * 2 * lbo_b, lbo_b, 128u);
#pragma unroll
                for (int m = 0; m < MT; m++) {
                  const uint64_t ad = umma_desc(
                      ta + static_cast<uint32_t>(ch * 8 + 2 * k) * S::kSlab + shift + m * 128u,
                      S::kSlab, S::kWp * 16u);
                  mma_bf16(d0 + m * a.NT, ad, bd, idesc, !first);
                }
                first = false;
              }
              if (!a.resident) mma_commit(&empty_b[sb]);
              if (++sb == a.stages_b) {
                sb = 0;
                pb ^= 1u;
              }
            }
          }
          if (!ok) break;
          mma_commit(&empty_a[sa]);
          if (++sa == a.stages_a) {
            sa = 0;
            pa ^= 1u;
          }
        }
        if (ok) mma_commit(&full_d[acc]);
      }
      if (!ok) {
        gave_up = 1;
        atomicExch(a.err, 1);
        int never = 0;
        mma_commit(&drained);  // the MMAs in flight end before the memory is given back
        mbar_wait(&drained, 0, &never);
      }
    }
  } else if (warp < 6) {
    // epilogue: lane = pixel of the tile's row group, 16 output channels at a time
    const int q = warp & 3;
    const int row = q * 32 + lane, py = row >> 3, px = row & 7;
    const int o0 = blockIdx.y * a.NT;
    int it = 0;
    for (int t = blockIdx.x; t < a.tiles; t += gridDim.x, it++) {
      const int acc = it & 1;
      if (!mbar_wait(&full_d[acc], (it >> 1) & 1, &gave_up)) {
        gave_up = 1;
        atomicExch(a.err, 1);
        break;
      }
      __syncwarp();
      fence_after();
      const int n = t / (a.tiles_x * a.tiles_y), r = t - n * (a.tiles_x * a.tiles_y);
      const int ty = r / a.tiles_x, tx = r - ty * a.tiles_x;
      const int i = ty * S::kH + py;
#pragma unroll
      for (int m = 0; m < MT; m++) {
        const int j = tx * S::kW + m * 8 + px;
        const bool in = i < a.H && j < a.W;
        const int64_t pix = in ? static_cast<int64_t>((n * a.H + i) * a.W + j) : 0;
        for (int c = 0; c < a.NT; c += 16) {
          uint32_t v[16];
          tmem_ld16(tmem + (static_cast<uint32_t>(q * 32) << 16) +
                        static_cast<uint32_t>((acc * MT + m) * a.NT + c),
                    v);
          tmem_wait_ld();
#pragma unroll
          for (int h = 0; h < 2; h++) {
            const int o = o0 + c + 8 * h;
            if (!in || o >= a.cos) continue;
            uint4 mk = make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
            if (a.mask) mk = *reinterpret_cast<const uint4 *>(a.mask + pix * a.cos + o);
            const uint32_t mw[4] = {mk.x, mk.y, mk.z, mk.w};
            uint32_t out[4];
#pragma unroll
            for (int e = 0; e < 8; e += 2) {
              __nv_bfloat16 w[2];
#pragma unroll
              for (int s = 0; s < 2; s++) {
                float f = __uint_as_float(v[8 * h + e + s]);
                const bool real = o + e + s < a.co;
                if (a.bias && real) f += a.bias[o + e + s];
                if (a.relu) f = fmaxf(f, 0.f);
                const __nv_bfloat16 mm = __ushort_as_bfloat16(
                    static_cast<unsigned short>(s ? mw[e / 2] >> 16 : mw[e / 2] & 0xFFFFu));
                if (!real || !(__bfloat162float(mm) > 0.f)) f = 0.f;
                w[s] = __float2bfloat16_rn(f);
                if (a.yf && real) a.yf[pix * a.co + o + e + s] = __bfloat162float(w[s]);
              }
              out[e / 2] = static_cast<uint32_t>(__bfloat16_as_ushort(w[0])) |
                           (static_cast<uint32_t>(__bfloat16_as_ushort(w[1])) << 16);
            }
            *reinterpret_cast<uint4 *>(a.y + pix * a.cos + o) =
                make_uint4(out[0], out[1], out[2], out[3]);
          }
        }
      }
      fence_before();
      mbar_arrive(&empty_d[acc]);
    }
  } else {
    // image tiles
    const int tid = threadIdx.x - 192;
    int sa = 0, it = 0;
    uint32_t pa = 0;
    bool ok = true;
    for (int t = blockIdx.x; ok && t < a.tiles; t += gridDim.x) {
      const int n = t / (a.tiles_x * a.tiles_y), r = t - n * (a.tiles_x * a.tiles_y);
      const int ty = r / a.tiles_x, tx = r - ty * a.tiles_x;
      const int i0 = ty * S::kH - S::kHalo, j0 = tx * S::kW - S::kHalo;
      const int units = a.parts * (KS * KS / a.unit_taps);
      for (int u = 0; u < units; u++, it++) {
        const int p = u % a.parts;
        if (it >= a.stages_a && !mbar_wait(&empty_a[sa], pa ^ 1u, &gave_up)) {
          ok = false;
          break;
        }
        const uint32_t dst = base_a + sa * stride_a;
        const int k8 = min(a.p8, a.k8 - p * a.p8);
        const uint32_t magic = p + 1 < a.parts ? a.magic : a.magic_last;
        for (int e = tid; e < S::kPix * k8; e += 128) {
          const int pix = static_cast<int>(__umulhi(static_cast<uint32_t>(e), magic));
          const int s8 = e - pix * k8, c8 = p * a.p8 + s8;
          const int y = pix / S::kWp, x = pix - y * S::kWp;
          const int i = i0 + y, j = j0 + x;
          const bool in = i >= 0 && i < a.H && j >= 0 && j < a.W && c8 < a.x.n8;
          cp_async16(dst + s8 * S::kSlab + pix * 16,
                     in ? input_at(a.x, n, i, j, a.H, a.W, c8) : a.x.xa, in);
        }
        cp_async_commit();
        if (a.stages_a == 1) {
          cp_async_wait<0>();
          fence_async_proxy();
          mbar_arrive(&full_a[sa]);
        } else if (it > 0) {  // the copies before these have landed
          cp_async_wait<1>();
          fence_async_proxy();
          mbar_arrive(&full_a[sa ? sa - 1 : a.stages_a - 1]);
        }
        if (++sa == a.stages_a) {
          sa = 0;
          pa ^= 1u;
        }
      }
    }
    cp_async_wait<0>();
    if (!ok) {
      gave_up = 1;
      atomicExch(a.err, 1);
    } else if (a.stages_a > 1 && it > 0) {
      fence_async_proxy();
      mbar_arrive(&full_a[sa ? sa - 1 : a.stages_a - 1]);
    }
  }
  __syncwarp();
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 1) tmem_dealloc(tmem, a.tmem_cols);
}

// ---------------------------------------------------------------------------
// Weight gradient
// ---------------------------------------------------------------------------
// dW[d][c][o] = sum_p X[p + d][c] gz[p][o]: per tap an accumulator with M =
// input channels (one block of 128), N = output channels (one block), K =
// pixels, 128 per stage (a tile of 8 x 16).  Both operands are MN-major
// views of the slabs, so nothing is transposed.  A CTA holds the
// accumulators of as many taps as tensor memory takes (a group) and sums one
// split of the tiles; the splits' sums go to `partials` and wgrad_reduce adds
// them in order (the same gradient every time).  The bias gradient is one
// more accumulator, whose X is all ones.
// kRep (few input channels): M = 3 x channels, the three horizontal taps of
// a row at once -- the tile is stored three times, shifted, and one
// accumulator per vertical tap remains.
constexpr int kWgThreads = 160;
constexpr int kWgStages = 3;

struct WgradDev {
  InputDev x;
  const __nv_bfloat16 *gz;
  int N, H, W, ci, ca, co, cos;   // ca: channels of the first source
  int NT, n_blocks;               // output-channel tile and how many
  int m_blocks, groups, group_taps;
  int tiles_x, tiles_y, tiles, splits;
  int stages;
  uint32_t tmem_cols;
  float *partials;
  int64_t len;                    // KS^2 ci co + co
  int *err;
};

template <int KS, bool kRep>
struct WgShape {
  static constexpr int kHalo = KS / 2;
  static constexpr int kWp = kRep ? 8 : 8 + 2 * kHalo, kHp = 16 + 2 * kHalo;
  static constexpr int kPixX = kWp * kHp;
  static constexpr uint32_t kSlabX = (kPixX | 1) * 16;
  static constexpr uint32_t kSlabG = 129 * 16;
  static constexpr uint32_t kBytesX = 16 * kSlabX;  // 128 channels
};

template <int KS, bool kRep>
__global__ void __launch_bounds__(kWgThreads, 1) wgrad_tc(const __grid_constant__ WgradDev a) {
  using S = WgShape<KS, kRep>;
  extern __shared__ __align__(128) unsigned char dyn[];
  __shared__ uint64_t full[kWgStages], empty[kWgStages], done;
  __shared__ uint32_t tmem_slot;
  __shared__ int gave_up;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
  const int n8g = a.NT / 8;
  const uint32_t stage_bytes = (S::kBytesX + n8g * S::kSlabG + 127u) & ~127u;
  const uint32_t ones = smem_addr(dyn), base = ones + 4096u;
  int job = blockIdx.x;
  const int nb = job % a.n_blocks;
  job /= a.n_blocks;
  const int mb = job % a.m_blocks, grp = job / a.m_blocks;
  const int o0 = nb * a.NT;
  // vertical taps (kRep) or taps of this group
  const int tap0 = grp * a.group_taps;
  const int ntap = min(a.group_taps, (kRep ? KS : KS * KS) - tap0);
  const bool with_bias = mb == 0 && grp == 0;
  // this split's tiles
  const int t0 = static_cast<int>(static_cast<int64_t>(a.tiles) * blockIdx.y / a.splits);
  const int t1 = static_cast<int>(static_cast<int64_t>(a.tiles) * (blockIdx.y + 1) / a.splits);
  if (tid == 0) {
    for (int i = 0; i < kWgStages; i++) {
      mbar_init(&full[i], 128);
      mbar_init(&empty[i], 1);
    }
    mbar_init(&done, 1);
    gave_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  for (int e = tid; e < 256; e += kWgThreads)
    *reinterpret_cast<uint4 *>(dyn + e * 16) =
        make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
  fence_async_proxy();
  if (warp == 4) tmem_alloc(&tmem_slot, a.tmem_cols);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_slot;

  if (warp == 4) {
    if (lane == 0) {
      const uint32_t idesc = umma_idesc(a.NT, true);
      bool ok = true;
      int st = 0;
      uint32_t ph = 0;
      for (int t = t0; t < t1; t++) {
        if (!mbar_wait(&full[st], ph, &gave_up)) {
          ok = false;
          break;
        }
        fence_after();
        const uint32_t sx = base + st * stage_bytes, sg = sx + S::kBytesX;
#pragma unroll 1
        for (int k = 0; k < 8; k++) {  // 16 pixels: two rows of the tile
          const uint64_t bd = umma_desc(sg + k * 256u, 128u, S::kSlabG);
          const bool acc = t > t0 || k > 0;
          for (int j = 0; j < ntap; j++) {
            const int tap = tap0 + j;
            const int dy = kRep ? tap : tap / KS, dx = kRep ? 0 : tap % KS;
            const uint64_t ad = umma_desc(
                sx + static_cast<uint32_t>((dy + 2 * k) * S::kWp + dx) * 16u, S::kWp * 16u,
                S::kSlabX);
            mma_bf16(tmem + j * a.NT, ad, bd, idesc, acc);
          }
          if (with_bias)
            mma_bf16(tmem + a.group_taps * a.NT, umma_desc(ones, 128u, 256u), bd, idesc, acc);
        }
        mma_commit(&empty[st]);
        if (++st == a.stages) {
          st = 0;
          ph ^= 1u;
        }
      }
      mma_commit(&done);
      if (!ok) {
        gave_up = 1;
        atomicExch(a.err, 1);
        int never = 0;
        mbar_wait(&done, 0, &never);
      }
    }
    __syncwarp();
  } else {
    // loads: this block's input slabs, then the gradient's
    const int n8x = min(16, a.x.n8 - mb * 16);
    const int units = kRep ? S::kHp * (8 + 2 * S::kHalo) * n8x : S::kPixX * n8x;
    constexpr int rowp = 8 + 2 * S::kHalo;
    // quotients by n8x and n8v (n8x may be 1: its reciprocal does not fit 32 bits)
    const uint32_t mx = n8x > 1 ? 0xFFFFFFFFu / static_cast<uint32_t>(n8x) + 1u : 0u;
    const int n8v = min(n8g, (a.cos - o0) / 8);
    const uint32_t mv = n8v > 1 ? 0xFFFFFFFFu / static_cast<uint32_t>(n8v) + 1u : 0u;
    bool ok = true;
    int st = 0, it = 0;
    uint32_t ph = 0;
    for (int t = t0; t < t1; t++, it++) {
      if (it >= a.stages && !mbar_wait(&empty[st], ph ^ 1u, &gave_up)) {
        ok = false;
        break;
      }
      const int n = t / (a.tiles_x * a.tiles_y), r = t - n * (a.tiles_x * a.tiles_y);
      const int ty = r / a.tiles_x, tx = r - ty * a.tiles_x;
      const uint32_t sx = base + st * stage_bytes, sg = sx + S::kBytesX;
      for (int e = tid; e < units; e += 128) {
        const int pix = n8x > 1 ? static_cast<int>(__umulhi(e, mx)) : e, c8 = e - pix * n8x;
        const int y = pix / rowp, x = pix - y * rowp;
        const int i = ty * 16 + y - S::kHalo, j = tx * 8 + x - S::kHalo;
        const bool in = i >= 0 && i < a.H && j >= 0 && j < a.W;
        const __nv_bfloat16 *src =
            in ? input_at(a.x, n, i, j, a.H, a.W, mb * 16 + c8) : a.x.xa;
        if constexpr (kRep) {
#pragma unroll
          for (int dx = 0; dx < KS; dx++)
            if (x >= dx && x < dx + 8)
              cp_async16(sx + (dx * n8x + c8) * S::kSlabX + (y * 8 + x - dx) * 16, src, in);
        } else {
          cp_async16(sx + c8 * S::kSlabX + pix * 16, src, in);
        }
      }
      for (int e = tid; e < 128 * n8v; e += 128) {
        const int pix = n8v > 1 ? static_cast<int>(__umulhi(e, mv)) : e, c8 = e - pix * n8v;
        const int i = ty * 16 + (pix >> 3), j = tx * 8 + (pix & 7);
        const bool in = i < a.H && j < a.W;
        cp_async16(sg + c8 * S::kSlabG + pix * 16,
                   in ? a.gz + static_cast<int64_t>((n * a.H + i) * a.W + j) * a.cos + o0 + c8 * 8
                      : a.gz,
                   in);
      }
      cp_async_commit();
      if (it > 0) {
        cp_async_wait<1>();
        fence_async_proxy();
        mbar_arrive(&full[st ? st - 1 : a.stages - 1]);
      }
      if (++st == a.stages) {
        st = 0;
        ph ^= 1u;
      }
    }
    cp_async_wait<0>();
    if (!ok) {
      gave_up = 1;
      atomicExch(a.err, 1);
    } else if (it > 0) {
      fence_async_proxy();
      mbar_arrive(&full[st ? st - 1 : a.stages - 1]);
    }
    // the sums of this split: lane = input channel (and horizontal tap)
    const bool have = ok && mbar_wait(&done, 0, &gave_up);
    if (!have) {
      gave_up = 1;
      atomicExch(a.err, 1);
    }
    __syncwarp();
    if (have) {
      fence_after();
      const bool empty_split = t1 <= t0;
      const int row = warp * 32 + lane;
      // row -> (dx, channel as the kernels see it) -> channel of the layer
      const int rows = n8x * 8;
      const int dxr = kRep ? row / rows : 0;
      const int cp = kRep ? row - dxr * rows : row;
      const int ck = mb * 128 + cp;  // padded channel
      const int ca8 = a.x.n8a * 8;
      const int c = ck < ca8 ? (ck < a.ca ? ck : -1)
                             : (a.ca + ck - ca8 < a.ci ? a.ca + ck - ca8 : -1);
      const bool valid = cp < rows && c >= 0 && (!kRep || dxr < KS);
      float *out = a.partials + static_cast<int64_t>(blockIdx.y) * a.len;
      const bool v4 = a.co % 4 == 0;
      for (int j = 0; j < ntap + (with_bias ? 1 : 0); j++) {
        const bool bias = j == ntap;
        const int col = bias ? a.group_taps : j;
        const int tap = kRep ? (tap0 + j) * KS + dxr : tap0 + j;
        float *dst = bias ? out + static_cast<int64_t>(KS * KS) * a.ci * a.co
                          : out + (static_cast<int64_t>(tap) * a.ci + c) * a.co;
        const bool write = bias ? row == 0 : valid;
        for (int cc = 0; cc < a.NT; cc += 16) {
          uint32_t v[16];
          tmem_ld16(tmem + (static_cast<uint32_t>(warp * 32) << 16) +
                        static_cast<uint32_t>(col * a.NT + cc),
                    v);
          tmem_wait_ld();
          if (!write) continue;
          const int o = o0 + cc;
#pragma unroll
          for (int e = 0; e < 16; e += 4) {
            float f[4];
#pragma unroll
            for (int s = 0; s < 4; s++) f[s] = empty_split ? 0.f : __uint_as_float(v[e + s]);
            if (v4) {
              if (o + e < a.co)
                *reinterpret_cast<float4 *>(dst + o + e) = make_float4(f[0], f[1], f[2], f[3]);
            } else {
#pragma unroll
              for (int s = 0; s < 4; s++)
                if (o + e + s < a.co) dst[o + e + s] = f[s];
            }
          }
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 4) tmem_dealloc(tmem, a.tmem_cols);
}

__global__ void __launch_bounds__(256) wgrad_reduce(const float *__restrict__ p, int splits,
                                                    int64_t len, float *__restrict__ out) {
  const int64_t e = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x;
  if (e >= len) return;
  float s = 0.f;
#pragma unroll 8
  for (int k = 0; k < splits; k++) s += p[k * len + e];
  out[e] = s;
}

// Packed weights: [output tile][tap][chunk of 64 channels][slab][output][8].
__global__ void __launch_bounds__(256) pack_kernel(const PackJob *__restrict__ jobs) {
  const PackJob J = jobs[blockIdx.y];
  const int KS2 = J.ks * J.ks, lci = J.ca + J.cb;
  // the packed convolution's inputs (two padded sources) and outputs
  const int ka = J.flip ? J.co : J.ca, kb = J.flip ? 0 : J.cb;
  const int k8 = pad16(pad8(ka) + pad8(kb)) / 8;
  // the adjoint's outputs are the layer's two inputs, padded the same way
  const int oa = J.flip ? J.ca : J.co, ob = J.flip ? J.cb : 0;
  const int co = J.flip ? pad8(J.ca) + pad8(J.cb) : J.co;
  const int NT = conv_tile_n(co);
  for (int64_t e = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x; e < J.elems;
       e += static_cast<int64_t>(gridDim.x) * 256) {
    const int sub = static_cast<int>(e & 7);
    int64_t q = e >> 3;
    const int o = static_cast<int>(q % NT);
    q /= NT;
    const int c8 = static_cast<int>(q % k8);
    q /= k8;
    const int d = static_cast<int>(q % KS2), nt = static_cast<int>(q / KS2);
    auto plain = [](int p, int a, int b) {  // padded index -> channel, or -1
      const int a8 = pad8(a);
      if (p < a8) return p < a ? p : -1;
      return p - a8 < b ? a + p - a8 : -1;
    };
    const int ki = plain(c8 * 8 + sub, ka, kb), oo = plain(nt * NT + o, oa, ob);
    float v = 0.f;
    if (ki >= 0 && oo >= 0)
      v = J.flip ? J.w[(static_cast<int64_t>(KS2 - 1 - d) * lci + oo) * J.co + ki]
                 : J.w[(static_cast<int64_t>(d) * lci + ki) * J.co + oo];
    J.out[e] = __float2bfloat16_rn(v);
  }
}

uint32_t pow2_cols(int c) {
  uint32_t p = 32;
  while (p < static_cast<uint32_t>(c)) p *= 2;
  return p;
}

InputDev input_dev(const ConvInput &in) {
  InputDev x;
  x.xa = in.xa;
  x.xb = in.xb;
  x.sa = pad8(in.ca);
  x.sb = pad8(in.cb);
  x.n8a = pad8(in.ca) / 8;
  x.n8 = in.padded() / 8;
  x.up = in.up;
  return x;
}

template <int KS, int MT>
cudaError_t conv_launch(ConvDev d, int sms, cudaStream_t s) {
  using S = TileShape<KS, MT>;
  const int n_blocks = (pad16(d.co) + d.NT - 1) / d.NT;
  d.tiles_x = (d.W + S::kW - 1) / S::kW;
  d.tiles_y = (d.H + S::kH - 1) / S::kH;
  d.tiles = d.N * d.tiles_x * d.tiles_y;
  const int gx = std::min(d.tiles, std::max(1, sms / n_blocks));
  const int per = (d.tiles + gx - 1) / gx;  // tiles a CTA walks over
  // input channels a tile takes at once: all, if one tile of them fits beside
  // three weight blocks
  const int b_bytes = d.NT * 128;
  const int fit = (kSmemMax - 3 * b_bytes) / static_cast<int>(S::kSlab) / 8 * 8;
  d.parts = d.k8 <= fit ? 1 : (d.k8 + fit - 1) / fit;
  d.p8 = d.parts == 1 ? d.k8 : fit;
  const int last = d.k8 - (d.parts - 1) * d.p8;
  d.magic = static_cast<uint32_t>((uint64_t(1) << 32) / d.p8 + 1);
  d.magic_last = static_cast<uint32_t>((uint64_t(1) << 32) / last + 1);
  const int sa_bytes = (d.p8 * static_cast<int>(S::kSlab) + 127) / 128 * 128;
  d.unit_taps = d.parts == 1 ? KS * KS : 1;
  const int blocks =
      KS * KS * ((d.parts - 1) * ((d.p8 + 7) / 8) + (last + 7) / 8);
  // all weights in shared memory where one image tile (two if there are
  // more) still fits beside them, else a ring of at least three blocks
  const int want_a = std::min(per * (d.parts == 1 ? 1 : d.parts * KS * KS), 2);
  d.resident = blocks <= kMaxStagesB && blocks * b_bytes + want_a * sa_bytes <= kSmemMax;
  d.stages_a = want_a;
  if (!d.resident && want_a * sa_bytes + 3 * b_bytes > kSmemMax) d.stages_a = 1;
  d.stages_b = d.resident ? blocks
                          : std::min({blocks, 8, (kSmemMax - d.stages_a * sa_bytes) / b_bytes});
  if (d.stages_b < 1) return cudaErrorInvalidValue;
  d.tmem_cols = pow2_cols(2 * MT * d.NT);
  // more than half of an SM's shared memory: one CTA per SM, so that its
  // tensor memory is the CTA's alone
  const int smem = std::max(d.stages_a * sa_bytes + d.stages_b * b_bytes, 120 * 1024);
  conv_halo_tc<KS, MT><<<dim3(gx, n_blocks), kConvThreads, smem, s>>>(d);
  return cudaGetLastError();
}

struct WgPlan {
  bool rep;
  int NT, n_blocks, m_blocks, groups, group_taps, splits, stages, tiles_x, tiles_y, tiles;
  uint32_t cols;
  int smem;
};
template <int KS, bool kRep>
void wg_smem(WgPlan *p) {
  using S = WgShape<KS, kRep>;
  const int stage = (static_cast<int>(S::kBytesX + p->NT / 8 * S::kSlabG) + 127) / 128 * 128;
  p->stages = std::min(kWgStages, (kSmemMax - 4096) / stage);
  p->smem = std::max(4096 + p->stages * stage, 120 * 1024);
}
WgPlan wg_plan(int ks, int ci_padded, int co, int N, int H, int W, int sms) {
  WgPlan p;
  p.rep = ks == 3 && 3 * ci_padded <= 128;
  p.NT = conv_tile_n(co);
  p.n_blocks = (pad16(co) + p.NT - 1) / p.NT;
  p.m_blocks = p.rep ? 1 : (ci_padded + 127) / 128;
  const int taps = p.rep ? ks : ks * ks;
  const int fit = std::max(1, 512 / p.NT - 1);  // accumulators beside the bias gradient's
  p.groups = (taps + fit - 1) / fit;
  p.group_taps = (taps + p.groups - 1) / p.groups;
  p.cols = pow2_cols((p.group_taps + 1) * p.NT);
  p.tiles_x = (W + 7) / 8;
  p.tiles_y = (H + 15) / 16;
  p.tiles = N * p.tiles_x * p.tiles_y;
  const int jobs = p.n_blocks * p.m_blocks * p.groups;
  p.splits = std::max(1, std::min(p.tiles, sms / jobs));
  if (ks == 3 && p.rep) wg_smem<3, true>(&p);
  else if (ks == 3) wg_smem<3, false>(&p);
  else wg_smem<1, false>(&p);
  return p;
}

}  // namespace

int64_t packed_elems(int ks, int ci_padded, int co) {
  const int NT = conv_tile_n(co);
  return static_cast<int64_t>((pad16(co) + NT - 1) / NT) * NT * ks * ks * pad16(ci_padded);
}

cudaError_t launch_pack(const PackJob *jobs_dev, int n_jobs, int64_t max_elems, cudaStream_t s) {
  const unsigned gx = static_cast<unsigned>(std::min<int64_t>(64, (max_elems + 2047) / 2048));
  pack_kernel<<<dim3(std::max(1u, gx), n_jobs), 256, 0, s>>>(jobs_dev);
  return cudaGetLastError();
}

cudaError_t setup_tc() {
  cudaError_t e = cudaSuccess;
  auto set = [&](auto *f) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
  };
  set(conv_halo_tc<3, 1>);
  set(conv_halo_tc<3, 2>);
  set(conv_halo_tc<1, 1>);
  set(conv_halo_tc<1, 2>);
  set(wgrad_tc<3, true>);
  set(wgrad_tc<3, false>);
  set(wgrad_tc<1, false>);
  return e;
}

cudaError_t launch_conv_tc(const ConvCall &c, int sms, int *err, cudaStream_t s) {
  ConvDev d{};
  d.x = input_dev(c.in);
  d.k8 = pad16(c.in.padded()) / 8;
  d.wk = c.wk;
  d.bias = c.bias;
  d.mask = c.mask;
  d.y = c.y;
  d.yf = c.yf;
  d.N = c.N;
  d.H = c.H;
  d.W = c.W;
  d.co = c.co;
  d.cos = pad8(c.co);
  d.NT = conv_tile_n(c.co);
  d.relu = c.relu;
  d.err = err;
  // two pixel blocks a tile halve the weights' traffic; one where two do not
  // fit beside three weight blocks, or would leave SMs without a tile
  const int tiles2 = c.N * ((c.W + 15) / 16) * ((c.H + 15) / 16);
  const int n_blocks = (pad16(c.co) + d.NT - 1) / d.NT;
  const int a2 = d.k8 * static_cast<int>(c.ks == 3 ? TileShape<3, 2>::kSlab : TileShape<1, 2>::kSlab);
  const bool two = a2 + 3 * d.NT * 128 <= kSmemMax && tiles2 * n_blocks >= sms;
  if (c.ks == 3) return two ? conv_launch<3, 2>(d, sms, s) : conv_launch<3, 1>(d, sms, s);
  return two ? conv_launch<1, 2>(d, sms, s) : conv_launch<1, 1>(d, sms, s);
}

int64_t wgrad_scratch(int ks, int ci, int ci_padded, int co, int N, int H, int W, int sms) {
  const WgPlan p = wg_plan(ks, ci_padded, co, N, H, W, sms);
  return static_cast<int64_t>(p.splits) * (static_cast<int64_t>(ks) * ks * ci * co + co);
}

cudaError_t launch_wgrad_tc(const ConvInput &in, int ks, const __nv_bfloat16 *gz, int co, int N,
                            int H, int W, float *partials, float *dw, int sms, int *err,
                            cudaStream_t s) {
  const WgPlan p = wg_plan(ks, in.padded(), co, N, H, W, sms);
  WgradDev d{};
  d.x = input_dev(in);
  d.gz = gz;
  d.N = N;
  d.H = H;
  d.W = W;
  d.ci = in.ca + in.cb;
  d.ca = in.ca;
  d.co = co;
  d.cos = pad8(co);
  d.NT = p.NT;
  d.n_blocks = p.n_blocks;
  d.m_blocks = p.m_blocks;
  d.groups = p.groups;
  d.group_taps = p.group_taps;
  d.tiles_x = p.tiles_x;
  d.tiles_y = p.tiles_y;
  d.tiles = p.tiles;
  d.splits = p.splits;
  d.stages = p.stages;
  d.tmem_cols = p.cols;
  d.partials = partials;
  d.len = static_cast<int64_t>(ks) * ks * d.ci * co + co;
  d.err = err;
  if (p.stages < 2) return cudaErrorInvalidValue;
  const dim3 grid(p.n_blocks * p.m_blocks * p.groups, p.splits);
  if (ks == 3 && p.rep) wgrad_tc<3, true><<<grid, kWgThreads, p.smem, s>>>(d);
  else if (ks == 3) wgrad_tc<3, false><<<grid, kWgThreads, p.smem, s>>>(d);
  else wgrad_tc<1, false><<<grid, kWgThreads, p.smem, s>>>(d);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  wgrad_reduce<<<static_cast<unsigned>((d.len + 255) / 256), 256, 0, s>>>(partials, p.splits, d.len,
                                                                           dw);
  return cudaGetLastError();
}

}  // namespace net
}  // namespace lbm
