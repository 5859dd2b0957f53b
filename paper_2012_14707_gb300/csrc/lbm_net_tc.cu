// Convolutions of the warm-start network's BF16 mode on the tcgen05 tensor
// cores: forward and backward-data (conv_halo_tc) and the weight gradient
// (wgrad_tc), with the packing of their weights.
//
// An image tile -- its pixels with the halo its taps reach -- is copied to
// shared memory once, and a tap's shifted operand is the same tile at another
// start address.  (Gathered per tap, nine times, the operands cost four
// times what the MMAs did: forward pass 256x256 x 8 images 3.23 ms, now 0.41;
// gradients 18.1 ms, now 1.62.)  Two layouts allow that:
// * conv_halo_tc: a 128-byte row of 64 channels per pixel, in the 128-byte
//   swizzle, which goes by address: row r's 16-byte unit u lies at unit u ^ (r
//   mod 8).  Channels are K (K-major).
// * wgrad_tc: "slabs" of 8 channels, 16 bytes per pixel, no swizzle: 8
//   neighbouring pixels of a slab are one core matrix, whatever pixel it
//   starts at.  Pixels are K (MN-major), so nothing is transposed.  A slab's
//   length is an odd number of 16-byte units, so the copies of a pixel's
//   slabs fall in different banks.
//
// What bounds them: an MMA of M = 128, K = 16 takes 54 cycles up to N = 64
// and 64 at N = 128 (measured, either layout), so the layers of 32 and 64
// output channels, 60 % of the network's flops, reach a quarter and a half of
// the tensor peak at best, and issuing the MMAs from one warp costs 70 to 100
// cycles each around that; but a tile's latency comes first: the MMAs of the
// forward pass take 145 of its 410 us (3 -> 32 channels: 6 of 32).  The channel
// order of the sums (taps outermost) is kept over all shapes, so results do
// not depend on them.
//
// Every wait is bounded; one that runs out sets *err, and the CTA's roles
// give up in turn after waiting for the copies they started.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "lbm_internal.h"
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
// Waits for the phase with parity `phase`; false if it did not come within
// kWaitLimit tries or the CTA gave up.  For a role that one lane runs.
// try_wait suspends the warp (for up to about the hint, a microsecond): warps
// polling with test_wait took so many issue slots that the roles with work to
// do ran several times slower (a 32-channel 256x256 layer 90 us).
constexpr int kWaitLimit = 1 << 20;
__device__ __forceinline__ bool mbar_wait_lane(uint64_t *bar, uint32_t phase,
                                               volatile int *gave_up) {
  const uint32_t a = smem_addr(bar);
  for (int it = 0; it < kWaitLimit; it++) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(a), "r"(phase), "r"(1000u)
        : "memory");
    if (done) return true;
    if ((it & 63) == 63 && *gave_up) return false;
  }
  return false;
}

// The same for a warp that waits as one: the answer is warp-uniform, so the
// loops around it are, and their counters and descriptors -- and no lane
// leaves alone ahead of a tcgen05 instruction that the whole warp executes.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t *bar, uint32_t phase,
                                               volatile int *gave_up) {
  return __all_sync(0xFFFFFFFFu, mbar_wait_lane(bar, phase, gave_up));
}

// Shared-memory matrix descriptor without swizzle; lbo, sbo in bytes.
// K-major operand: lbo between core matrices along K, sbo between groups of
// 8 rows.  MN-major operand: sbo between core matrices along M (N), lbo
// between groups of 8 along K.  Bit 46: descriptor version.
// The low word holds the address and lbo, so a descriptor further on in the
// same tile is the low word plus the distance / 16: one addition per MMA
// (the issuing thread is alone; 64-bit descriptor arithmetic cost it 150 to
// 240 cycles an MMA, several times what the MMA takes).
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lbo) {
  return ((addr >> 4) & 0x3FFFu) | (((lbo >> 4) & 0x3FFFu) << 16);
}
constexpr uint32_t kSwizzle128 = 2u << 29;  // layout type, high word
__device__ __forceinline__ uint32_t desc_hi(uint32_t sbo) {
  return ((sbo >> 4) & 0x3FFFu) | (1u << 14);
}
// kind::f16, D = FP32, A = B = BF16, M = 128; mn: both operands MN-major
__host__ __device__ constexpr uint32_t umma_idesc(int N, bool mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (mn ? (1u << 15) | (1u << 16) : 0u) |
         (static_cast<uint32_t>(N >> 3) << 17) | (static_cast<uint32_t>(128 >> 4) << 24);
}
// The MMA warp runs its loops with all lanes, and one lane (leader != 0)
// issues: descriptors and loop counters are then warp-uniform, as the
// instruction takes them.
__device__ __forceinline__ uint32_t elect_leader() {
  uint32_t l;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xFFFFFFFF;\n selp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(l));
  return l;
}
__device__ __forceinline__ void mma_bf16(uint32_t leader, uint32_t d, uint32_t alo, uint32_t ahi,
                                         uint32_t blo, uint32_t bhi, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p, q;\n .reg .b64 a, b;\n setp.ne.b32 p, %6, 0;\n setp.ne.b32 q, %7, 0;\n"
      " mov.b64 a, {%1, %2};\n mov.b64 b, {%3, %4};\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n}\n" ::"r"(d),
      "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(accumulate), "r"(leader)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t leader, uint64_t *bar) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
      " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(
          smem_addr(bar)),
      "r"(leader)
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
// p = v (set) or p += v in FP32, rounded to nearest, without waiting for it
__device__ __forceinline__ void add_or_set(float *p, const float (&v)[4], bool set) {
  if (set)
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
  else
    asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"l"(p),
                 "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3])
                 : "memory");
}
__device__ __forceinline__ void add_or_set(float *p, float v, bool set) {
  if (set)
    *p = v;
  else
    asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;\n" ::"l"(p), "f"(v) : "memory");
}
// v[r] (of each of 4 neighbouring lanes: the lane's r-th quarter) becomes the
// lane's own quarter of the r-th of them: the four then write a row together
__device__ __forceinline__ void transpose4(float (&v)[4][4], int lane) {
#pragma unroll
  for (int x = 1; x < 4; x *= 2) {
    const bool up = lane & x;
#pragma unroll
    for (int r = 0; r < 4; r++) {
      if (r & x) continue;
#pragma unroll
      for (int s = 0; s < 4; s++) {
        const float got = __shfl_xor_sync(0xFFFFFFFFu, up ? v[r][s] : v[r + x][s], x);
        if (up) v[r][s] = got;
        else v[r + x][s] = got;
      }
    }
  }
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
// Arrives at *bar (one of its expected arrivals) once this thread's copies so
// far have landed; the thread goes on at once.
__device__ __forceinline__ void cp_async_arrive(uint64_t *bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];\n" ::"r"(smem_addr(bar))
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_all;\n" ::: "memory");
}
// Waits until the kernels before this one in the stream are complete, then
// lets the next one start its CTAs as this one's finish (launch_chained).
// Packed weights and biases, which no kernel of a pass writes, may be read
// before it.
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
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

// Both sources of a convolution's input, in slabs (groups of 8 channels).
struct InputDev {
  const __nv_bfloat16 *xa, *xb;
  int sa, sb;        // pixel strides (elements)
  int n8a, n8;       // slabs of xa, of both
  int up;
};
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
// eight warps copy image tiles (cp.async, zero outside the image), one lane
// issues the MMAs (M = 128 pixels, N = NT, K = 16), eight warps read the
// accumulators back, of which there are two sets, so that a tile's epilogue
// overlaps the next tile's MMAs.
constexpr int kLoadThreads = 256;
constexpr int kConvThreads = 320 + kLoadThreads;
constexpr int kMaxStagesB = 54;   // 9 taps x 6 chunks of 64: every weight block resident
constexpr int kMaxStagesA = 2;
constexpr int kSmemMax = 232448 - 2048;  // dynamic shared memory a CTA may use (static below)

struct ConvDev {
  InputDev x;
  int k8;                 // slabs the MMAs run over (even; those >= x.n8 are zero)
  // ... in `parts` parts of p8 slabs, as many as shared memory takes at once;
  // one part: a tile is copied once for all taps; more: again for every tap
  int parts, p8, unit_taps;
  int lanes_log2;         // threads of the image copy that share a pixel
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
  // 64 channels of the tile: a row of 128 bytes per pixel, in whole swizzle
  // patterns of 1024 bytes
  static constexpr uint32_t kChunk = (kPix * 128 + 1023) / 1024 * 1024;
};

template <int KS, int MT>
__global__ void __launch_bounds__(kConvThreads, 1) conv_halo_tc(const __grid_constant__ ConvDev a) {
  using S = TileShape<KS, MT>;
  extern __shared__ __align__(128) unsigned char dyn[];
  __shared__ uint64_t full_a[kMaxStagesA], empty_a[kMaxStagesA];
  __shared__ uint64_t full_b[kMaxStagesB], empty_b[kMaxStagesB];
  __shared__ uint64_t full_d[2], empty_d[2], drained;
  __shared__ __align__(16) float bias[128];
  __shared__ uint32_t tmem_slot;
  __shared__ int gave_up;
  const int warp = __shfl_sync(0xFFFFFFFFu, static_cast<int>(threadIdx.x >> 5), 0);
  const int lane = threadIdx.x & 31;
  const uint32_t stride_a = static_cast<uint32_t>((a.p8 + 7) / 8) * S::kChunk;
  const uint32_t b_bytes = static_cast<uint32_t>(a.NT) * 128u;  // 64 channels
  const uint32_t base_a = (smem_addr(dyn) + 1023u) & ~1023u;
  const uint32_t base_b = base_a + static_cast<uint32_t>(a.stages_a) * stride_a;
  if (threadIdx.x == 0) {
    for (int i = 0; i < a.stages_a; i++) {
      mbar_init(&full_a[i], kLoadThreads);
      mbar_init(&empty_a[i], 1);
    }
    for (int i = 0; i < a.stages_b; i++) {
      mbar_init(&full_b[i], 1);
      mbar_init(&empty_b[i], 1);
    }
    for (int i = 0; i < 2; i++) {
      mbar_init(&full_d[i], 1);
      mbar_init(&empty_d[i], 256);
    }
    mbar_init(&drained, 1);
    gave_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (threadIdx.x >= 64 && threadIdx.x < 64 + a.NT) {
    const int o = blockIdx.y * a.NT + threadIdx.x - 64;
    bias[threadIdx.x - 64] = a.bias && o < a.co ? a.bias[o] : 0.f;
  }
  if (warp == 1) tmem_alloc(&tmem_slot, a.tmem_cols);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, tmem_slot, 0);

  if (warp != 0) chain_wait();
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
            // the ring's first blocks are copied while the kernel before
            // runs; the bounded wait for a free block starts after it, when
            // the MMAs do
            if (issued == a.stages_b) chain_wait();
            if (issued >= a.stages_b && !mbar_wait_lane(&empty_b[st], ph ^ 1u, &gave_up)) {
              ok = false;
              break;
            }
            const int tap = t0 + b / chunks, c8 = (b % chunks) * 8;
            const uint32_t bytes = static_cast<uint32_t>(min(8, k8 - c8)) * a.NT * 16u;
            const int64_t at = static_cast<int64_t>(tap * a.k8 + p * a.p8 + c8) * a.NT * 16;
            mbar_expect(&full_b[st], bytes);
            bulk_copy(base_b + (a.resident ? static_cast<uint32_t>(at) : st * b_bytes), src + at,
                      bytes, &full_b[st]);
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
          mbar_wait_lane(&full_b[i % a.stages_b], (i / a.stages_b) & 1, &never);
      }
    }
  } else if (warp == 1) {
    // MMAs
    const uint32_t leader = elect_leader();
    const uint32_t idesc = umma_idesc(a.NT, false);
    const uint32_t lbo_b = static_cast<uint32_t>(a.NT) * 16u;
    const uint32_t ahi = desc_hi(S::kWp * 128u) | kSwizzle128, bhi = desc_hi(128u);
    const uint32_t step_b = 2 * lbo_b / 16;
    int sa = 0, sb = 0, it = 0;
    uint32_t pa = 0, pb = 0;
    bool ok = true;
    for (int t = blockIdx.x; ok && t < a.tiles; t += gridDim.x, it++) {
      const int acc = it & 1;
      if (it >= 2 && !mbar_wait_warp(&empty_d[acc], ((it >> 1) & 1) ^ 1u, &gave_up)) {
        ok = false;
        break;
      }
      const uint32_t d0 = tmem + static_cast<uint32_t>(acc * MT * a.NT);
      const bool wait_b = !a.resident || it == 0;  // resident weights land once
      if (a.resident) {
        sb = 0;
        pb = 0;
      }
      uint32_t accumulate = 0, b_at = 0;
      // the MMAs of one tap of a tile in shared memory
      auto do_tap = [&](uint32_t alo, int k8) {
#pragma unroll 1
        for (int c8 = 0; c8 < k8; c8 += 8, alo += S::kChunk / 16 - 8u) {
          if (wait_b) {
            if (!mbar_wait_warp(&full_b[sb], pb, &gave_up)) {
              ok = false;
              return;
            }
            fence_after();
          }
          // resident blocks lie end to end, a ring's at its stride
          uint32_t blo = desc_lo(base_b, lbo_b) + (a.resident ? b_at : sb * (b_bytes / 16));
          const int k16 = min(4, (k8 - c8) >> 1);
          b_at += static_cast<uint32_t>(k16) * step_b;
#pragma unroll 1
          for (int k = 0; k < k16; k++) {
#pragma unroll
            for (int m = 0; m < MT; m++)
              mma_bf16(leader, d0 + m * a.NT, alo + m * 64u, ahi, blo, bhi, idesc, accumulate);
            accumulate = 1;
            alo += 2;  // 16 channels on
            blo += step_b;
          }
          if (!a.resident) mma_commit(leader, &empty_b[sb]);
          if (++sb == a.stages_b) {
            sb = 0;
            pb ^= 1u;
          }
        }
      };
      auto next_tile = [&](uint32_t *ta) {
        if (!mbar_wait_warp(&full_a[sa], pa, &gave_up)) {
          ok = false;
          return;
        }
        fence_async_proxy();  // the landed copies, for the MMAs
        fence_after();
        *ta = desc_lo(base_a + sa * stride_a, 16u);
      };
      auto free_tile = [&]() {
        mma_commit(leader, &empty_a[sa]);
        if (++sa == a.stages_a) {
          sa = 0;
          pa ^= 1u;
        }
      };
      uint32_t ta = 0;
      if (a.parts == 1) {
        next_tile(&ta);
        if (!ok) break;
        // (rolled: nine copies of the body would miss the instruction cache)
        int dx = 0;
#pragma unroll 1
        for (int tap = 0; tap < KS * KS; tap++) {
          do_tap(ta, a.k8);
          if (!ok) break;
          ta += 8;
          if (++dx == KS) {
            dx = 0;
            ta += (S::kWp - KS) * 8;
          }
        }
        if (!ok) break;
        free_tile();
      } else {
        for (int tap = 0; ok && tap < KS * KS; tap++)
          for (int p = 0; ok && p < a.parts; p++) {
            next_tile(&ta);
            if (!ok) break;
            do_tap(ta + ((tap / KS) * S::kWp + (tap % KS)) * 8, min(a.p8, a.k8 - p * a.p8));
            if (ok) free_tile();
          }
        if (!ok) break;
      }
      mma_commit(leader, &full_d[acc]);
    }
    if (!ok) {
      gave_up = 1;
      if (lane == 0) atomicExch(a.err, 1);
      int never = 0;
      mma_commit(leader, &drained);  // the MMAs in flight end before the memory is given back
      mbar_wait_warp(&drained, 0, &never);
    }
  } else if (warp < 10) {
    // epilogue: lane = pixel of a block; the two groups of four warps take a
    // pixel block each (MT = 2) or alternate channel groups (MT = 1); 16
    // output channels at a time
    const int q = warp & 3, grp = (warp - 2) >> 2;
    const int row = q * 32 + lane, py = row >> 3, px = row & 7;
    const int m = MT == 2 ? grp : 0;
    const int c_first = MT == 2 ? 0 : grp * 16, c_step = MT == 2 ? 16 : 32;
    const int o0 = blockIdx.y * a.NT;
    int it = 0;
    for (int t = blockIdx.x; t < a.tiles; t += gridDim.x, it++) {
      const int acc = it & 1;
      const int n = t / (a.tiles_x * a.tiles_y), r = t - n * (a.tiles_x * a.tiles_y);
      const int ty = r / a.tiles_x, tx = r - ty * a.tiles_x;
      const int i = ty * S::kH + py, j = tx * S::kW + m * 8 + px;
      const bool in = i < a.H && j < a.W;
      const int64_t pix = in ? static_cast<int64_t>((n * a.H + i) * a.W + j) : 0;
      if (!mbar_wait_warp(&full_d[acc], (it >> 1) & 1, &gave_up)) {
        gave_up = 1;
        if (lane == 0) atomicExch(a.err, 1);
        break;
      }
      fence_after();
      const uint32_t col = tmem + (static_cast<uint32_t>(q * 32) << 16) +
                           static_cast<uint32_t>((acc * MT + m) * a.NT);
      for (int c = c_first; c < a.NT; c += c_step) {
        const int o = o0 + c;
        const bool st0 = in && o < a.cos, st1 = in && o + 8 < a.cos;
        uint4 mk[2];
        if (a.mask) {
          const uint4 *mp = reinterpret_cast<const uint4 *>(a.mask + pix * a.cos + o);
          if (st0) mk[0] = mp[0];
          if (st1) mk[1] = mp[1];
        }
        uint32_t v[16];
        tmem_ld16(col + c, v);
        tmem_wait_ld();
        // channels beyond the layer's have zero weights and bias: zeros
        float f[16];
#pragma unroll
        for (int e = 0; e < 16; e += 4) {
          const float4 b4 = *reinterpret_cast<const float4 *>(&bias[c + e]);
          f[e] = __uint_as_float(v[e]) + b4.x;
          f[e + 1] = __uint_as_float(v[e + 1]) + b4.y;
          f[e + 2] = __uint_as_float(v[e + 2]) + b4.z;
          f[e + 3] = __uint_as_float(v[e + 3]) + b4.w;
        }
        if (a.relu) {
#pragma unroll
          for (int e = 0; e < 16; e++) f[e] = fmaxf(f[e], 0.f);
        }
        uint32_t w[8];
#pragma unroll
        for (int e = 0; e < 8; e++) {
          const __nv_bfloat162 b2 = __floats2bfloat162_rn(f[2 * e], f[2 * e + 1]);
          w[e] = *reinterpret_cast<const uint32_t *>(&b2);
        }
        if (a.mask) {
          const uint32_t g[8] = {mk[0].x, mk[0].y, mk[0].z, mk[0].w,
                                 mk[1].x, mk[1].y, mk[1].z, mk[1].w};
#pragma unroll
          for (int e = 0; e < 8; e++) {
            if (!(__uint_as_float(g[e] << 16) > 0.f)) w[e] &= 0xFFFF0000u;
            if (!(__uint_as_float(g[e] & 0xFFFF0000u) > 0.f)) w[e] &= 0xFFFFu;
          }
        }
        uint4 *yp = reinterpret_cast<uint4 *>(a.y + pix * a.cos + o);
        if (st0) yp[0] = make_uint4(w[0], w[1], w[2], w[3]);
        if (st1) yp[1] = make_uint4(w[4], w[5], w[6], w[7]);
        if (a.yf && in) {
#pragma unroll
          for (int e = 0; e < 16; e++)
            if (o + e < a.co)
              a.yf[pix * a.co + o + e] =
                  __uint_as_float(e & 1 ? w[e / 2] & 0xFFFF0000u : w[e / 2] << 16);
        }
      }
      fence_before();
      mbar_arrive(&empty_d[acc]);
    }
  } else {
    // image tiles
    // lane groups of `lanes` threads copy neighbouring slabs of a pixel (the
    // power of two that divides a part's slabs), then the slabs `lanes` on;
    // a thread's pixels are `pstep` apart, so its coordinates advance by
    // additions
    const int tid = threadIdx.x - 320;
    const int lanes = 1 << a.lanes_log2, g8 = tid & (lanes - 1);
    const int pix0 = tid >> a.lanes_log2, pstep = kLoadThreads >> a.lanes_log2;
    const int dy = pstep / S::kWp, dx = pstep - dy * S::kWp;
    const int y0 = pix0 / S::kWp, x0 = pix0 - y0 * S::kWp;
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
        if (it >= a.stages_a && !mbar_wait_warp(&empty_a[sa], pa ^ 1u, &gave_up)) {
          ok = false;
          break;
        }
        const int k8 = min(a.p8, a.k8 - p * a.p8);
        int y = y0, x = x0;
        const uint32_t dst = base_a + sa * stride_a;
        const int Wa = a.W >> a.x.up, rows = n * (a.H >> a.x.up);
        const int first = (n * a.H + i0) * a.W + j0, c0 = p * a.p8 + g8;
        const bool plain = !a.x.up && a.x.n8 == a.x.n8a;  // one source at full resolution
        for (int pix = pix0; pix < S::kPix; pix += pstep) {
          const int i = i0 + y, j = j0 + x;
          const bool in = static_cast<unsigned>(i) < static_cast<unsigned>(a.H) &&
                          static_cast<unsigned>(j) < static_cast<unsigned>(a.W);
          const int here = first + y * a.W + x;
          const __nv_bfloat16 *pa8 = a.x.xa, *pb8 = a.x.xa;
          if (in) {
            pa8 += static_cast<int64_t>(plain ? here
                                              : (rows + (i >> a.x.up)) * Wa + (j >> a.x.up)) *
                       a.x.sa +
                   c0 * 8;
            if (!plain) pb8 = a.x.xb + static_cast<int64_t>(here) * a.x.sb + (c0 - a.x.n8a) * 8;
          }
          for (int s8 = g8; s8 < k8; s8 += lanes) {
            const int c8 = p * a.p8 + s8;
            const bool valid = in && c8 < a.x.n8;
            cp_async16(dst + (s8 >> 3) * S::kChunk + pix * 128 + (((s8 ^ pix) & 7) << 4),
                       valid ? (c8 < a.x.n8a ? pa8 : pb8) + (s8 - g8) * 8 : a.x.xa, valid);
          }
          y += dy;
          x += dx;
          if (x >= S::kWp) {
            x -= S::kWp;
            y++;
          }
        }
        cp_async_arrive(&full_a[sa]);
        if (++sa == a.stages_a) {
          sa = 0;
          pa ^= 1u;
        }
      }
    }
    cp_async_wait_all();
    if (!ok) {
      gave_up = 1;
      if (lane == 0) atomicExch(a.err, 1);
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
// The accumulators hold FP32, but the tensor cores truncate as they add: a sum
// is biased towards zero by half a unit in the last place of its size per
// MMA.  So an accumulator runs over kWgChain tiles (512 pixels, 32 MMAs) at
// most; then eight warps read it and add it, rounding to nearest, to the
// split's sums in memory, tap by tap, while the next chain's MMAs follow.
// Relative error of the gradients of positive operands (base 32 and 64,
// 256x256 x 8) for chains without limit, of 6, 4 and 3 tiles: 7.6e-6 and
// 2.2e-5, 6.9e-7 and 7.5e-7, 3.6e-7 and 3.7e-7, 2.6e-7; gradients of the
// 256x256 x 8 network 1414, 1484, 1542, 1602 us.
// kRep (few input channels): M = 3 x channels, the three horizontal taps of
// a row at once -- the tile is stored three times, shifted, and one
// accumulator per vertical tap remains.
constexpr int kWgLoaders = 256;
constexpr int kWgDrain = 256;  // threads that read the sums back
constexpr int kWgChain = 4;    // tiles an accumulator runs over, at most
constexpr int kWgThreads = kWgLoaders + 32 + kWgDrain;
constexpr int kWgStages = 3;

struct WgradDev {
  InputDev x;
  const __nv_bfloat16 *gz;
  int N, H, W, ci, ca, co, cos;   // ca: channels of the first source
  int NT, n_blocks;               // output-channel tile and how many
  int m_blocks, groups, group_taps;
  int tiles_x, tiles_y, tiles, splits;
  int stages;
  int lanes_x, lanes_g;           // log2 of the threads that share a pixel's copies
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
  __shared__ uint64_t full[kWgStages], empty[kWgStages];
  __shared__ uint64_t done, drained[10];  // a chain's sums; read back, per tap (9: the bias)
  __shared__ uint32_t tmem_slot;
  __shared__ int gave_up;
  const int warp = __shfl_sync(0xFFFFFFFFu, static_cast<int>(threadIdx.x >> 5), 0);
  const int lane = threadIdx.x & 31, tid = threadIdx.x;
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
  // ... in as few chains as kWgChain allows, all about as long
  const int fewest = (t1 - t0 + kWgChain - 1) / kWgChain;
  const int per_chain = (t1 - t0 + fewest - 1) / fewest;
  if (tid == 0) {
    for (int i = 0; i < kWgStages; i++) {
      mbar_init(&full[i], kWgLoaders);
      mbar_init(&empty[i], 1);
    }
    mbar_init(&done, 1);
    for (int i = 0; i < 9; i++) mbar_init(&drained[i], kWgDrain);
    mbar_init(&drained[9], 32);
    gave_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  for (int e = tid; e < 256; e += kWgThreads)
    *reinterpret_cast<uint4 *>(dyn + e * 16) =
        make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
  fence_async_proxy();
  if (warp == 8) tmem_alloc(&tmem_slot, a.tmem_cols);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, tmem_slot, 0);

  chain_wait();
  if (warp == 8) {
    const uint32_t leader = elect_leader();
    const uint32_t idesc = umma_idesc(a.NT, true);
    const uint32_t ahi = desc_hi(S::kSlabX), bhi = desc_hi(S::kSlabG);
    const uint32_t ones_lo = desc_lo(ones, 128u), ones_hi = desc_hi(256u);
    const uint32_t bias_d = tmem + a.group_taps * a.NT;
    bool ok = true;
    int st = 0, chain = 0, left = 0;  // chains committed, tiles left of this one
    uint32_t ph = 0;
    for (int t = t0; t < t1; t++) {
      if (!mbar_wait_warp(&full[st], ph, &gave_up)) {
        ok = false;
        break;
      }
      fence_async_proxy();  // the landed copies, for the MMAs
      fence_after();
      const uint32_t sx = base + st * stage_bytes;
      // 16 pixels (two rows of the tile) per MMA
      uint32_t xlo = desc_lo(sx, S::kWp * 16u);
      uint32_t glo = desc_lo(sx + S::kBytesX, 128u);
      if (left == 0 && chain > 0) {
        // a further chain's first tile goes tap by tap (the bias last), each
        // as soon as the sums of the chain before have been read
#pragma unroll 1
        for (int j = 0; j < ntap + (with_bias ? 1 : 0); j++) {
          const bool bias = j == ntap;
          if (!mbar_wait_warp(&drained[bias ? 9 : j], (chain - 1) & 1, &gave_up)) {
            ok = false;
            break;
          }
          fence_after();
          const int tap = tap0 + j;
          const uint32_t d = bias ? bias_d : tmem + j * a.NT;
          const uint32_t alo = bias ? ones_lo
                                    : xlo + (kRep ? tap * S::kWp : (tap / KS) * S::kWp + tap % KS);
#pragma unroll 1
          for (int k = 0; k < 8; k++)
            mma_bf16(leader, d, alo + (bias ? 0 : k * 2 * S::kWp), bias ? ones_hi : ahi,
                     glo + 16 * k, bhi, idesc, k);
        }
        if (!ok) break;
      } else {
#pragma unroll 1
        for (int k = 0; k < 8; k++) {
          // taps tap0 .. tap0 + ntap - 1 (vertical taps where kRep)
          const uint32_t acc = left != 0 || k != 0;
#pragma unroll
          for (int tap = 0; tap < (kRep ? KS : KS * KS); tap++) {
            const int j = tap - tap0;
            if (j >= 0 && j < ntap)
              mma_bf16(leader, tmem + j * a.NT,
                       xlo + (kRep ? tap * S::kWp : (tap / KS) * S::kWp + tap % KS), ahi, glo, bhi,
                       idesc, acc);
          }
          if (with_bias) mma_bf16(leader, bias_d, ones_lo, ones_hi, glo, bhi, idesc, acc);
          xlo += 2 * S::kWp;
          glo += 16;
        }
      }
      if (left == 0) left = min(per_chain, t1 - t);
      mma_commit(leader, &empty[st]);
      if (++st == a.stages) {
        st = 0;
        ph ^= 1u;
      }
      if (--left == 0) {
        mma_commit(leader, &done);
        chain++;
      }
    }
    if (!ok) {
      gave_up = 1;
      if (lane == 0) atomicExch(a.err, 1);
      // the MMAs in flight end before the memory is given back
      int never = 0;
      if (chain > 0) mbar_wait_warp(&done, (chain - 1) & 1, &never);
      mma_commit(leader, &done);
      mbar_wait_warp(&done, chain & 1, &never);
    }
    __syncwarp();
  } else if (warp < 8) {
    // loads: this block's input slabs, then the gradient's
    const int n8x = min(16, a.x.n8 - mb * 16);
    constexpr int kPix = S::kHp * (8 + 2 * S::kHalo);
    constexpr int rowp = 8 + 2 * S::kHalo;
    const int n8v = min(n8g, (a.cos - o0) / 8);
    // as in conv_halo_tc: `lanes` threads share a pixel
    const int lx = 1 << a.lanes_x, gx8 = tid & (lx - 1), px0 = tid >> a.lanes_x,
              pxs = kWgLoaders >> a.lanes_x;
    const int ly = 1 << a.lanes_g, gg8 = tid & (ly - 1), pg0 = tid >> a.lanes_g,
              pgs = kWgLoaders >> a.lanes_g;
    const int dyx = pxs / rowp, dxx = pxs - dyx * rowp;
    const int yx0 = px0 / rowp, xx0 = px0 - yx0 * rowp;
    // this block's slabs of the first source, and which sources it reads
    const int n8xa = a.x.n8a - mb * 16;
    const bool use_a = n8xa > 0, use_b = n8xa < n8x;
    const uint32_t rep_stride = static_cast<uint32_t>(n8x) * S::kSlabX;
    bool ok = true;
    int st = 0, it = 0;
    uint32_t ph = 0;
    for (int t = t0; t < t1; t++, it++) {
      if (it >= a.stages && !mbar_wait_warp(&empty[st], ph ^ 1u, &gave_up)) {
        ok = false;
        break;
      }
      const int n = t / (a.tiles_x * a.tiles_y), r = t - n * (a.tiles_x * a.tiles_y);
      const int ty = r / a.tiles_x, tx = r - ty * a.tiles_x;
      const uint32_t sx = base + st * stage_bytes, sg = sx + S::kBytesX;
      const int i0 = ty * 16 - S::kHalo, j0 = tx * 8 - S::kHalo;
      const int first = (n * a.H + i0) * a.W + j0, rows = n * (a.H >> a.x.up);
      constexpr int kBatch = kRep ? 1 : 4;  // pixels whose addresses are formed together
      int y = yx0, x = xx0;
      for (int pix = px0; pix < kPix; pix += kBatch * pxs) {
        const __nv_bfloat16 *pa8[kBatch], *pb8[kBatch];
        bool in[kBatch];
        int at[kBatch], xq[kBatch];
#pragma unroll
        for (int q = 0; q < kBatch; q++) {
          in[q] = static_cast<unsigned>(i0 + y) < static_cast<unsigned>(a.H) &&
                  static_cast<unsigned>(j0 + x) < static_cast<unsigned>(a.W);
          pa8[q] = a.x.xa;
          pb8[q] = a.x.xa;
          const int here = first + y * a.W + x;
          if (in[q]) {
            if (use_a)
              pa8[q] += static_cast<int64_t>(a.x.up ? (rows + ((i0 + y) >> 1)) * (a.W >> 1) +
                                                          ((j0 + x) >> 1)
                                                    : here) *
                            a.x.sa +
                        mb * 128;
            if (use_b)
              pb8[q] = a.x.xb + static_cast<int64_t>(here) * a.x.sb + (mb * 16 - a.x.n8a) * 8;
          }
          at[q] = kRep ? (y * 8 + x) * 16 : (pix + q * pxs) * 16;
          xq[q] = x;
          y += dyx;
          x += dxx;
          if (x >= rowp) {
            x -= rowp;
            y++;
          }
        }
        for (int s8 = gx8; s8 < n8x; s8 += lx) {
#pragma unroll
          for (int q = 0; q < kBatch; q++) {
            if (pix + q * pxs >= kPix) continue;
            const __nv_bfloat16 *src = in[q] ? (s8 < n8xa ? pa8[q] : pb8[q]) + s8 * 8 : a.x.xa;
            const uint32_t d = sx + s8 * S::kSlabX + at[q];
            if constexpr (kRep) {
#pragma unroll
              for (int dx = 0; dx < KS; dx++)
                if (static_cast<unsigned>(xq[q] - dx) < 8u)
                  cp_async16(d + dx * rep_stride - dx * 16, src, in[q]);
            } else {
              cp_async16(d, src, in[q]);
            }
          }
        }
      }
#pragma unroll 4
      for (int pix = pg0; pix < 128; pix += pgs) {
        const int i = ty * 16 + (pix >> 3), j = tx * 8 + (pix & 7);
        const bool in = i < a.H && j < a.W;
        const __nv_bfloat16 *src =
            in ? a.gz + static_cast<int64_t>((n * a.H + i) * a.W + j) * a.cos + o0 : a.gz;
        for (int s8 = gg8; s8 < n8v; s8 += ly)
          cp_async16(sg + s8 * S::kSlabG + pix * 16, in ? src + s8 * 8 : a.gz, in);
      }
      cp_async_arrive(&full[st]);
      if (++st == a.stages) {
        st = 0;
        ph ^= 1u;
      }
    }
    cp_async_wait_all();
    if (!ok) {
      gave_up = 1;
      if (lane == 0) atomicExch(a.err, 1);
    }
  } else {
    // the sums of each chain: lane = input channel (and horizontal tap), a
    // tap's blocks of 16 outputs in turn for the two groups of four warps
    const int q = warp & 3, row = q * 32 + lane, half = (warp - 9) >> 2;
    // row -> (dx, channel as the kernels see it) -> channel of the layer
    const int rows = min(16, a.x.n8 - mb * 16) * 8;
    const int dxr = kRep ? row / rows : 0;
    const int cp = kRep ? row - dxr * rows : row;
    const int ck = mb * 128 + cp;  // padded channel
    const int ca8 = a.x.n8a * 8;
    const int c = ck < ca8 ? (ck < a.ca ? ck : -1)
                           : (a.ca + ck - ca8 < a.ci ? a.ca + ck - ca8 : -1);
    const bool valid = cp < rows && c >= 0 && (!kRep || dxr < KS);
    // the row's place among a tap's (a row of taps') sums, or -1; and those of
    // the four rows that four neighbouring lanes write together
    const int at = valid ? (dxr * a.ci + c) * a.co : -1;
    int at4[4];
#pragma unroll
    for (int r = 0; r < 4; r++) at4[r] = __shfl_sync(0xFFFFFFFFu, at, (lane & ~3) + r);
    float *out = a.partials + static_cast<int64_t>(blockIdx.y) * a.len;
    const bool v4 = a.co % 4 == 0;
    for (int ch = 0; ch * per_chain < t1 - t0; ch++) {
      if (!mbar_wait_warp(&done, ch & 1, &gave_up)) {
        gave_up = 1;
        if (lane == 0) atomicExch(a.err, 1);
        break;
      }
      fence_after();
      for (int j = 0; j < ntap; j++) {
        float *dst = out + static_cast<int64_t>(tap0 + j) * (kRep ? KS : 1) * a.ci * a.co + o0;
        for (int cc = 16 * ((half + j * (a.NT / 16)) & 1); cc < a.NT; cc += 64) {
          float v[2][4][4];
          const bool two = cc + 32 < a.NT;
          const uint32_t at0 = tmem + (static_cast<uint32_t>(q * 32) << 16) +
                               static_cast<uint32_t>(j * a.NT + cc);
          tmem_ld16(at0, reinterpret_cast<uint32_t (&)[16]>(v[0]));
          if (two) tmem_ld16(at0 + 32, reinterpret_cast<uint32_t (&)[16]>(v[1]));
          tmem_wait_ld();
          if (cc + 64 >= a.NT) {
            fence_before();
            mbar_arrive(&drained[j]);
          }
#pragma unroll
          for (int h = 0; h < 2; h++) {
            if (h == 1 && !two) break;
            if (v4) {
              transpose4(v[h], lane);
              const int o = cc + 32 * h + 4 * (lane & 3);
#pragma unroll
              for (int r = 0; r < 4; r++)
                if (at4[r] >= 0 && o0 + o < a.co) add_or_set(dst + at4[r] + o, v[h][r], ch == 0);
            } else {
#pragma unroll
              for (int e = 0; e < 16; e++)
                if (at >= 0 && o0 + cc + 32 * h + e < a.co)
                  add_or_set(dst + at + cc + 32 * h + e, v[h][e / 4][e % 4], ch == 0);
            }
          }
          __syncwarp();
        }
        // (a half without a block of this tap)
        if (16 * ((half + j * (a.NT / 16)) & 1) >= a.NT) mbar_arrive(&drained[j]);
      }
      if (with_bias && warp == 12) {  // every row holds it
        for (int cc = 0; cc < a.NT; cc += 16) {
          uint32_t v[16];
          tmem_ld16(tmem + static_cast<uint32_t>(a.group_taps * a.NT + cc), v);
          tmem_wait_ld();
          float mine = 0.f;
#pragma unroll
          for (int e = 0; e < 16; e++)
            if (lane == e) mine = __uint_as_float(v[e]);
          if (lane < 16 && o0 + cc + lane < a.co)
            add_or_set(out + static_cast<int64_t>(KS * KS) * a.ci * a.co + o0 + cc + lane, mine,
                       ch == 0);
          __syncwarp();
        }
        fence_before();
        mbar_arrive(&drained[9]);
      }
    }
  }
  __syncwarp();
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 8) tmem_dealloc(tmem, a.tmem_cols);
}

// Sums the splits in a fixed order: group g of a CTA's G groups of threads
// adds splits g, g + G, ... of its 256 / G outputs, then the groups' sums are
// added in turn.  Many splits of few outputs need the groups to fill the GPU
// (152 splits of 9 k outputs: 14 us with one group, 7 with eight), few splits
// of many outputs lose by them (12 of 590 k: 10 against 24 us).
template <int G>
__global__ void __launch_bounds__(256) wgrad_reduce(const float *p, int splits, int64_t len,
                                                    float *out) {
  constexpr int kOut = 256 / G;
  __shared__ float sh[G][kOut];
  chain_wait();
  const int g = threadIdx.x / kOut, o = threadIdx.x % kOut;
  const int64_t e = static_cast<int64_t>(blockIdx.x) * kOut + o;
  float s = 0.f;
  if (e < len) {
#pragma unroll 4
    for (int k = g; k < splits; k += G) s += p[k * len + e];
  }
  if constexpr (G > 1) {
    sh[g][o] = s;
    __syncthreads();
    if (g == 0)
      for (int k = 1; k < G; k++) s += sh[k][o];
  }
  if (g == 0 && e < len) out[e] = s;
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
  const int fit = (kSmemMax - 1024 - 3 * b_bytes) / static_cast<int>(S::kChunk) * 8;
  d.parts = d.k8 <= fit ? 1 : (d.k8 + fit - 1) / fit;
  d.p8 = d.parts == 1 ? d.k8 : fit;
  const int last = d.k8 - (d.parts - 1) * d.p8;
  d.lanes_log2 = 1;  // both are even
  while (d.lanes_log2 < 3 && (d.p8 >> d.lanes_log2) % 2 == 0 && (last >> d.lanes_log2) % 2 == 0)
    d.lanes_log2++;
  const int sa_bytes = (d.p8 + 7) / 8 * static_cast<int>(S::kChunk);
  d.unit_taps = d.parts == 1 ? KS * KS : 1;
  const int blocks =
      KS * KS * ((d.parts - 1) * ((d.p8 + 7) / 8) + (last + 7) / 8);
  // all weights in shared memory where one image tile (two if there are
  // more) still fits beside them, else a ring of at least three blocks
  const int want_a = std::min(per * (d.parts == 1 ? 1 : d.parts * KS * KS), 2);
  // (their blocks end to end; parts of the channels never are)
  const int all_b = KS * KS * d.k8 * d.NT * 16;
  d.resident = d.parts == 1 && blocks <= kMaxStagesB &&
               all_b + want_a * sa_bytes <= kSmemMax - 1024;
  d.stages_a = want_a;
  if (!d.resident && want_a * sa_bytes + 3 * b_bytes > kSmemMax - 1024) d.stages_a = 1;
  d.stages_b = d.resident ? blocks
                          : std::min({blocks, 8, (kSmemMax - 1024 - d.stages_a * sa_bytes) / b_bytes});
  if (d.stages_b < 1) return cudaErrorInvalidValue;
  d.tmem_cols = pow2_cols(2 * MT * d.NT);
  // where the CTA takes more than half of tensor memory: more than half of
  // shared memory too, so that no other CTA waits beside it
  const int smem = std::max(1024 + d.stages_a * sa_bytes +
                                (d.resident ? all_b : d.stages_b * b_bytes),
                            d.tmem_cols > 256 ? 120 * 1024 : 0);
  return launch_chained(conv_halo_tc<KS, MT>, dim3(gx, n_blocks), kConvThreads, smem, s, d);
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
  p->smem = std::max(4096 + p->stages * stage, p->cols > 256 ? 120 * 1024 : 0);
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
  const int a2 = (d.k8 + 7) / 8 *
                 static_cast<int>(c.ks == 3 ? TileShape<3, 2>::kChunk : TileShape<1, 2>::kChunk);
  const bool two = a2 + 3 * d.NT * 128 <= kSmemMax - 1024 && tiles2 * n_blocks >= sms;
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
  // as many threads as a block has slabs, at most 16, as a power of two
  auto log2_floor = [](int v) {
    int l = 0;
    while (l < 4 && (2 << l) <= v) l++;
    return l;
  };
  d.lanes_x = log2_floor(std::min(16, in.padded() / 8));
  d.lanes_g = log2_floor(std::min(p.NT, d.cos) / 8);
  d.partials = partials;
  d.len = static_cast<int64_t>(ks) * ks * d.ci * co + co;
  d.err = err;
  if (p.stages < 2) return cudaErrorInvalidValue;
  const dim3 grid(p.n_blocks * p.m_blocks * p.groups, p.splits);
  cudaError_t e = ks != 3 ? launch_chained(wgrad_tc<1, false>, grid, kWgThreads, p.smem, s, d)
                  : p.rep ? launch_chained(wgrad_tc<3, true>, grid, kWgThreads, p.smem, s, d)
                          : launch_chained(wgrad_tc<3, false>, grid, kWgThreads, p.smem, s, d);
  if (e != cudaSuccess) return e;
  auto reduce = [&](auto groups) {
    constexpr int G = decltype(groups)::value;
    return launch_chained(wgrad_reduce<G>,
                          dim3(static_cast<unsigned>((d.len + 256 / G - 1) / (256 / G))), 256, 0, s,
                          static_cast<const float *>(partials), p.splits, d.len, dw);
  };
  if (p.splits >= 64) return reduce(std::integral_constant<int, 8>());
  if (p.splits >= 32) return reduce(std::integral_constant<int, 2>());
  return reduce(std::integral_constant<int, 1>());
}

}  // namespace net
}  // namespace lbm
