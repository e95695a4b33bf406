// 3x3 / stride 2 / padding 1 convolutions of the proposal network: the data
// gradients of layers 3-6 (dgrad_tma_kernel, below) and the forward passes
// (layers 2-4: NHWC bfloat16 maps 60x80x32 -> 30x40x64 -> 15x20x128 ->
// 8x10x256) on the 5th-generation tensor cores with TMA-fed operands.
//
// One CTA computes an output tile of 128 pixels (TH rows x TW columns of one
// image) for all C_out channels as a 128 x C_out x (9 C_in) product: one
// tcgen05.mma (M = 128, N = C_out, K = 16, bf16 x bf16 -> f32 in tensor
// memory) per tap and 16 input channels.  Its operands come straight from
// tiled TMA loads, no gather in software:
//  * A (im2col rows): for tap (ky, kx) and KB channels (KB = 32 or 64, a
//    64- or 128-byte row per pixel), a box of the input map {KB channels,
//    2 TW columns, 2 TH rows} starting at input pixel (2 ox0 + kx - 1,
//    2 oy0 + ky - 1) with element stride 2 in both pixel dimensions loads
//    the TH x TW input pixels that tap reads -- zero-filled where the
//    padding lies (negative or past-the-edge coordinates).  In shared memory
//    output pixel m's KB channels are row m, written with the TMA's 64- or
//    128-byte swizzle: the K-major swizzled layout tcgen05 reads (8-row
//    atoms of 8 x KB x 2 bytes), the K steps of 16 channels 32 bytes apart
//    inside a row.
//  * B (weights [C_out][9 C_in], K = tap x C_in + channel): a box {KB k,
//    C_out rows} in the same swizzled K-major layout.
// One warp issues the loads S stages ahead (mbarrier transaction counts),
// another the MMAs; a stage is refilled once the tcgen05.commit of the MMAs
// that read it has arrived.  Four warps read the accumulator back (tcgen05.ld)
// and apply bias, ReLU and the bfloat16 rounding of the other kernels.
// Every wait is bounded: past the limit the kernel records an error in
// *err, stops issuing, waits (bounded) for what it issued and frees its
// tensor memory.  Layers 5 and 6 (4 x 5 and 2 x 3 outputs) put several whole
// images in one tile: a box's fourth dimension spans them.  Layers 3 and 4
// at large batches use a persistent, warp-specialised form with two TMEM
// accumulators (conv_tma_pers_kernel).
#include <cuda.h>
#include <cuda_bf16.h>

#include <mutex>

#include "conv_tma.h"
#include "gs2d_common.cuh"
#include "per_device.h"

namespace gs2d {
namespace net {
namespace {

using bf16 = __nv_bfloat16;
constexpr int kConvThreads = 128;
constexpr int kWaitSpins = 1 << 24;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity) {
  for (int i = 0; i < kWaitSpins; ++i) {
    uint32_t ok;
    asm volatile(
        "{.reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;}\n"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    if (ok) return true;
  }
  return false;
}
// Shared-memory matrix descriptor of a K-major operand with rows of SW bytes
// (64 or 128) under the matching swizzle: start address, leading offset 16
// bytes (unused by the swizzled K-major layouts), stride 8 x SW bytes
// between the 8-row atoms, swizzle mode in bits 61-63 (2 = 128 B, 4 = 64 B).
template <int SW>
__device__ __forceinline__ uint64_t sw_desc(uint32_t saddr) {
  constexpr uint64_t mode = SW == 128 ? 2ull : 4ull;
  return (uint64_t)((saddr >> 4) & 0x3FFF) | (1ull << 16) |
         ((uint64_t)(((8 * SW) >> 4) & 0x3FFF) << 32) | (1ull << 46) | (mode << 61);
}
// Descriptor of an operand that is contiguous along its M / N dimension, in
// 128-byte rows of 64 elements (a row per k) under the 128-byte swizzle:
// leading offset mn_step between blocks of 64 elements, stride 1024 bytes
// between groups of 8 k.
__device__ __forceinline__ uint64_t mn_desc(uint32_t saddr, uint32_t mn_step) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((mn_step >> 4) & 0x3FFF) << 16) |
         ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// Instruction descriptor of kind::f16: f32 accumulate, bf16 A and B, A
// K-major, B K-major or contiguous along N, N = n, M = 128.
__host__ __device__ constexpr uint32_t mma_idesc(int n, bool b_mn = false) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (b_mn ? 1u << 16 : 0u) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(128 >> 4) << 24);
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int c0, int c1,
                                            int c2, int c3, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, "
      "{%2, %3, %4, %5}], [%6];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int c0, int c1,
                                            int c2, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, "
      "{%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int c0, int c1,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, "
      "{%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}

// A tile is NI images' TW x TH output pixels (a 128-pixel part of one image,
// or whole small images, TW x TH = the output map) times NB of the
// C_out channels.  One box per tap and channel block spans the NI images
// (its fourth dimension), so image g's pixels are rows [g TW TH, (g + 1) TW TH)
// of the 128-row MMA tile; rows past NI TW TH hold stale data whose results
// the epilogue drops.
template <int CIN, int COUT, int HI, int WI, int TW, int TH, int S, int NI = 1, int NB = COUT>
struct ConvTma {
  static constexpr int HO = (HI + 1) / 2, WO = (WI + 1) / 2;
  static constexpr int TX = (WO + TW - 1) / TW, TY = (HO + TH - 1) / TH;
  static constexpr int KB = CIN < 64 ? CIN : 64;  // channels per box row
  static constexpr int SW = KB * 2;               // row bytes = swizzle span
  static constexpr int CB = CIN / KB;             // boxes (stages) per tap
  static constexpr int KS = 9 * CB;               // stages per tile
  static constexpr int MMAS = KB / 16;            // MMAs per stage
  static constexpr int ROWS = NI * TW * TH;       // rows one input box lands
  static constexpr int BOX_BYTES = ROWS * SW;     // one input box (NI images)
  static constexpr int A_BYTES = 128 * SW;        // the 128-row A operand
  static constexpr int B_BYTES = NB * SW;         // one weight box
  static constexpr int STAGE = A_BYTES + B_BYTES;
  static constexpr int TX_BYTES = BOX_BYTES + B_BYTES;  // bytes a stage's loads bring
  static constexpr int SMEM = S * STAGE + 1024;   // + slack for 1024-byte alignment
  static constexpr int TMEM_COLS = NB;
  static constexpr int NSPLIT = COUT / NB;        // channel groups (grid.y)
  static constexpr bool B_MN = false;             // weights K-major
  static constexpr int B_STEP = 32;               // bytes from one K step of 16 to the next
  static __device__ __forceinline__ uint64_t b_desc(uint32_t saddr) { return sw_desc<SW>(saddr); }
  static_assert((NI == 1 && TW * TH == 128) || (TX == 1 && TY == 1 && ROWS <= 128),
                "one 128-row MMA tile: a part of one image, or whole images");
  static_assert(KB == 32 || KB == 64, "64- or 128-byte swizzled rows");
  static_assert(CIN % KB == 0 && NB >= 32 && NB <= 256 && (NB & (NB - 1)) == 0 &&
                    COUT % NB == 0,
                "tensor-memory columns: a power of two in [32, 256]");
  static_assert(A_BYTES % 1024 == 0 && B_BYTES % 1024 == 0, "swizzle atoms stay aligned");
  static_assert(2 * TW <= 256 && 2 * TH <= 256, "TMA box dimensions");
};

// The two issuing roles of a tile, each a whole warp whose lane 0 issues: the
// loop counters, barrier addresses and descriptors are then warp-uniform, and
// only the issuing instructions are predicated.  As single-thread loops with
// a descriptor built per MMA they took ~0.5 us per K step (of 9 to 36),
// whatever the step's bytes and MMAs, and were most of a small batch's time.

// Commit of every MMA issued so far to barrier bar, by lane 0.
__device__ __forceinline__ void commit_lane0(uint32_t bar) {
  asm volatile(
      "{.reg .pred q; setp.eq.u32 q, %1, 0;\n"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];}\n" ::"r"(bar),
      "r"(threadIdx.x & 31)
      : "memory");
}

// K steps 0 .. steps - 1 of one tile into the accumulator at tmem, the stages'
// running number starting at g0.  False when a wait ran out (the steps before
// it are issued).
template <class C, int S, int N>
__device__ __forceinline__ bool mma_steps(uint32_t tmem, int g0, int steps, const uint64_t* s_full,
                                          const uint64_t* s_empty, uint32_t stages,
                                          volatile int* s_consumed) {
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t a0 = sw_desc<C::SW>(stages), b0 = C::b_desc(stages + C::A_BYTES);
  const uint32_t a_lo = (uint32_t)a0, a_hi = (uint32_t)(a0 >> 32);
  const uint32_t b_lo = (uint32_t)b0, b_hi = (uint32_t)(b0 >> 32);
  int st = g0 % S;
  uint32_t phase = (uint32_t)((g0 / S) & 1);
#pragma unroll 1
  for (int s = 0; s < steps; ++s) {
    if (!bar_wait(smem_u32(s_full + st), phase)) return false;
    *s_consumed = g0 + s + 1;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // the address field counts 16 bytes and does not carry out of its 14 bits
    const uint32_t off = (uint32_t)st * (C::STAGE / 16);
#pragma unroll
    for (int j = 0; j < C::MMAS; ++j) {
      // K step j of the stage: 16 channels, 32 bytes into every swizzled row
      // (or 16 rows of 128 bytes)
      asm volatile(
          "{.reg .pred p, q; .reg .b64 da, db;\n"
          "setp.ne.b32 p, %6, 0; setp.eq.u32 q, %7, 0;\n"
          "mov.b64 da, {%1, %2}; mov.b64 db, {%3, %4};\n"
          "@q tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;}\n" ::"r"(tmem),
          "r"(a_lo + off + 2 * j), "r"(a_hi), "r"(b_lo + off + (C::B_STEP / 16) * j), "r"(b_hi),
          "r"(mma_idesc(N, C::B_MN)), "r"((s > 0 || j > 0) ? 1u : 0u), "r"(lane));
    }
    commit_lane0(smem_u32(s_empty + st));
    if (++st == S) {
      st = 0;
      phase ^= 1u;
    }
  }
  return true;
}

// Loads of `steps` K steps (KS per tile), a stage's once the MMAs that read
// its previous fill are done.  origin(tile step, x, y, n): the input pixel of
// tap (0, 0) and the image of the tile that step s belongs to.
template <class C, int CIN, int S, class Origin>
__device__ __forceinline__ void load_steps(const CUtensorMap& map_x, const CUtensorMap& map_w,
                                           int steps, const uint64_t* s_full,
                                           const uint64_t* s_empty, uint32_t stages,
                                           volatile int* s_issued, int* s_fail, Origin origin,
                                           int nb0) {
  const uint32_t lane = threadIdx.x & 31;
  int st = 0, x = 0, y = 0, n = 0, cb = 0, kx = 0, ky = 0, k = 0;
  uint32_t phase = 1u;   // of the stage's previous fill
#pragma unroll 1
  for (int g = 0; g < steps; ++g) {
    if (k == 0) origin(g, x, y, n);
    if (g >= S && !bar_wait(smem_u32(s_empty + st), phase)) {
      if (lane == 0) atomicExch(s_fail, 1);
      return;
    }
    const uint32_t base = stages + (uint32_t)st * C::STAGE;
    if (lane == 0) {
      const uint32_t bar = smem_u32(s_full + st);
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                   "r"(C::TX_BYTES)
                   : "memory");
      tma_load_4d(base, &map_x, cb, x + kx, y + ky, n, bar);
      tma_load_2d(base + C::A_BYTES, &map_w, (3 * ky + kx) * CIN + cb, nb0, bar);
    }
    *s_issued = g + 1;
    // next channel block, tap, tile
    cb += C::KB;
    if (cb == CIN) {
      cb = 0;
      if (++kx == 3) {
        kx = 0;
        if (++ky == 3) ky = 0;
      }
    }
    if (++k == C::KS) k = 0;
    if (++st == S) {
      st = 0;
      phase ^= 1u;
    }
  }
}

template <int CIN, int COUT, int HI, int WI, int TW, int TH, int S, int NI, int NB>
__global__ void __launch_bounds__(kConvThreads) conv_tma_kernel(
    const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
    const float* __restrict__ bias, bf16* __restrict__ out, int B, int* __restrict__ err) {
  using C = ConvTma<CIN, COUT, HI, WI, TW, TH, S, NI, NB>;
  extern __shared__ unsigned char conv_raw[];
  __shared__ __align__(8) uint64_t s_full[S], s_empty[S], s_done;
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail, s_issued, s_consumed;
  unsigned char* stages = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(conv_raw) + 1023) & ~(uintptr_t)1023);
  const int tile = blockIdx.x;
  // NI == 1: tile -> (image, TH x TW part); NI > 1: images tile NI .. tile NI + NI - 1
  const int img = NI == 1 ? tile / (C::TX * C::TY) : tile * NI;
  const int r = NI == 1 ? tile % (C::TX * C::TY) : 0;
  const int oy0 = (r / C::TX) * TH, ox0 = (r % C::TX) * TW;
  const int nb0 = (int)blockIdx.y * NB;  // first output channel of the tile
  const int warp = threadIdx.x >> 5;

  if (threadIdx.x == 0) {
    s_fail = 0;
    s_issued = 0;
    s_consumed = 0;
    for (int i = 0; i < S; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_full[i])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_empty[i])));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_done)));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&s_tmem)),
                 "r"(C::TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s_tmem;

  // warp 1 issues every load, warp 0 every MMA, so that the MMAs wait for
  // nothing but their operands
  if (warp == 1)
    load_steps<C, CIN, S>(map_x, map_w, C::KS, s_full, s_empty, smem_u32(stages), &s_issued,
                          &s_fail, [&](int s, int& x, int& y, int& n) {
                            (void)s;
                            x = 2 * ox0 - 1;
                            y = 2 * oy0 - 1;
                            n = img;   // images past the batch read as zeros
                          }, nb0);
  if (warp == 0) {
    const int ok = mma_steps<C, S, NB>(tmem, 0, C::KS, s_full, s_empty, smem_u32(stages), &s_consumed);
    // one last commit tracks every MMA issued (all, or those before a failure)
    commit_lane0(smem_u32(&s_done));
    if (!ok) s_fail = 1;
  }
  if (!bar_wait(smem_u32(&s_done), 0u)) atomicExch(&s_fail, 1);
  __syncthreads();
  // loads issued but not consumed (after a failure) land before the CTA exits
  if (threadIdx.x == 32)
    for (int s = s_consumed; s < s_issued; ++s)
      bar_wait(smem_u32(&s_full[s % S]), (uint32_t)((s / S) & 1));
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (!*reinterpret_cast<volatile int*>(&s_fail)) {
    // TMEM lane = row m: image img + m / (TW TH), output pixel (oy0 + q / TW,
    // ox0 + q % TW) with q = m % (TW TH)
    const int m = threadIdx.x;
    const int g = m / (TW * TH), q = m % (TW * TH);
    const int oy = oy0 + q / TW, ox = ox0 + q % TW;
    const bool ok = g < NI && img + g < B && oy < C::HO && ox < C::WO;
    bf16* dst = out + (((size_t)(img + g) * C::HO + oy) * C::WO + ox) * COUT + nb0;
    const float* bs = bias + nb0;
#pragma unroll 1
    for (int c0 = 0; c0 < NB; c0 += 16) {
      uint32_t v[16];
      const uint32_t taddr = tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)c0;
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, "
          "%10, %11, %12, %13, %14, %15}, [%16];\n"
          : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
            "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
            "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
          : "r"(taddr));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      if (ok) {
        uint32_t packed[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float x0 = fmaxf(__uint_as_float(v[2 * j]) + bs[c0 + 2 * j], 0.f);
          const float x1 = fmaxf(__uint_as_float(v[2 * j + 1]) + bs[c0 + 2 * j + 1], 0.f);
          const __nv_bfloat162 b2 = __floats2bfloat162_rn(x0, x1);
          packed[j] = *reinterpret_cast<const uint32_t*>(&b2);
        }
        uint4* d = reinterpret_cast<uint4*>(dst + c0);
        d[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
        d[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
      }
    }
  } else if (threadIdx.x == 0 && err) {
    atomicExch(err, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(C::TMEM_COLS));
}

// Persistent form for grids of many tiles (layers 2-4 at large batches):
// each CTA walks tiles blockIdx.x, blockIdx.x + gridDim.x, ... with three
// roles -- warp 4 issues the TMA loads S stages ahead across tile boundaries,
// warp 5 issues the MMAs into one of two TMEM accumulators, warps 0-3 read
// the other accumulator back -- so a tile's epilogue overlaps the next
// tile's loads and MMAs, and barrier set-up and TMEM allocation happen once
// per CTA.  Barriers: full/empty per stage (loads <-> MMAs), tfull/tempty
// per accumulator (MMAs <-> epilogue; tempty takes one arrival per epilogue
// warp).  Every tile sums its K steps in the same order as conv_tma_kernel,
// so results do not depend on the form or the grid.  Waits are bounded; a
// role whose wait runs out records the failure and stops; the MMA issuer's
// last commit tracks every MMA issued and all threads wait for it before
// the tensor memory is freed, and the loader waits for its loads in flight.
constexpr int kPersThreads = 192;

template <int CIN, int COUT, int HI, int WI, int TW, int TH, int S>
__global__ void __launch_bounds__(kPersThreads) conv_tma_pers_kernel(
    const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
    const float* __restrict__ bias, bf16* __restrict__ out, int n_tiles, int* __restrict__ err) {
  using C = ConvTma<CIN, COUT, HI, WI, TW, TH, S>;
  extern __shared__ unsigned char conv_raw[];
  __shared__ __align__(8) uint64_t s_full[S], s_empty[S], s_tfull[2], s_tempty[2], s_done;
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail, s_issued, s_consumed;
  unsigned char* stages = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(conv_raw) + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int my_n = (int)blockIdx.x < n_tiles
                       ? (n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x
                       : 0;
  if (threadIdx.x == 0) {
    s_fail = 0;
    s_issued = 0;
    s_consumed = 0;
    for (int i = 0; i < S; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_full[i])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_empty[i])));
    }
    for (int b = 0; b < 2; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_tfull[b])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 4;" ::"r"(smem_u32(&s_tempty[b])));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_done)));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&s_tmem)),
                 "r"(2 * C::TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s_tmem;

  if (warp == 4) {
    load_steps<C, CIN, S>(map_x, map_w, my_n * C::KS, s_full, s_empty, smem_u32(stages), &s_issued,
                          &s_fail, [&](int g, int& x, int& y, int& n) {
                            const int tile = (int)blockIdx.x + g / C::KS * (int)gridDim.x;
                            const int r = tile % (C::TX * C::TY);
                            n = tile / (C::TX * C::TY);
                            x = 2 * (r % C::TX) * TW - 1;
                            y = 2 * (r / C::TX) * TH - 1;
                          }, 0);
  } else if (warp == 5) {
    bool ok = true;
    for (int k = 0; k < my_n && ok; ++k) {
      const int buf = k & 1;
      // the epilogue has read this accumulator's previous tile
      if (k >= 2 && !bar_wait(smem_u32(&s_tempty[buf]), (uint32_t)(((k >> 1) - 1) & 1))) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      ok = mma_steps<C, S, COUT>(tmem + (uint32_t)(buf * C::TMEM_COLS), k * C::KS, C::KS, s_full, s_empty,
                                 smem_u32(stages), &s_consumed);
      if (ok) commit_lane0(smem_u32(&s_tfull[buf]));
    }
    // one last commit tracks every MMA issued
    commit_lane0(smem_u32(&s_done));
    if (!ok && lane == 0) atomicExch(&s_fail, 1);
  } else {
    // warps 0-3: TMEM lane = row m = threadIdx.x = output pixel (oy0 + m / TW, ox0 + m % TW)
    const int m = threadIdx.x;
    for (int k = 0; k < my_n; ++k) {
      const int buf = k & 1;
      if (!bar_wait(smem_u32(&s_tfull[buf]), (uint32_t)((k >> 1) & 1))) {
        atomicExch(&s_fail, 1);
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int tile = (int)blockIdx.x + k * (int)gridDim.x;
      const int img = tile / (C::TX * C::TY), r = tile % (C::TX * C::TY);
      const int oy = (r / C::TX) * TH + m / TW, ox = (r % C::TX) * TW + m % TW;
      const bool ok = oy < C::HO && ox < C::WO;
      bf16* dst = out + (((size_t)img * C::HO + oy) * C::WO + ox) * COUT;
#pragma unroll 1
      for (int c0 = 0; c0 < COUT; c0 += 16) {
        uint32_t v[16];
        const uint32_t taddr =
            tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)(buf * C::TMEM_COLS + c0);
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, "
            "%10, %11, %12, %13, %14, %15}, [%16];\n"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
              "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
              "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
            : "r"(taddr));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (ok) {
          uint32_t packed[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float x0 = fmaxf(__uint_as_float(v[2 * j]) + bias[c0 + 2 * j], 0.f);
            const float x1 = fmaxf(__uint_as_float(v[2 * j + 1]) + bias[c0 + 2 * j + 1], 0.f);
            const __nv_bfloat162 b2 = __floats2bfloat162_rn(x0, x1);
            packed[j] = *reinterpret_cast<const uint32_t*>(&b2);
          }
          uint4* d = reinterpret_cast<uint4*>(dst + c0);
          d[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
          d[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
        }
      }
      // this accumulator may be overwritten once all four warps have read it
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&s_tempty[buf]))
                     : "memory");
    }
  }
  __syncthreads();
  // every MMA issued has completed before the tensor memory is freed, and
  // loads issued but not consumed (after a failure) land before the CTA exits
  if (!bar_wait(smem_u32(&s_done), 0u)) atomicExch(&s_fail, 1);
  if (warp == 4 && lane == 0)
    for (int g = s_consumed; g < s_issued; ++g)
      bar_wait(smem_u32(&s_full[g % S]), (uint32_t)((g / S) & 1));
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && s_fail && err) atomicExch(err, 1);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(2 * C::TMEM_COLS));
}

// Data gradient of a layer (3-6): dx = mask * (dz convolved with the
// transposed weights), by parity class (py, px) of the input pixels (iy, ix)
// = (2 cy + py, 2 cx + px).  A class sees the taps ky = 1 (py = 0) or 0 and 2
// (py = 1), likewise in x, and under one tap its pixels read neighbouring
// pixels of dz at the offset (py && ky == 0, px && kx == 0): a plain box of
// dz, zeros past the edge.  So the product of a class tile (TH x TW class
// pixels of one image, or NI whole images) with NB input channels is, per tap
// and 64 output channels, one A box {64 channels, TW, TH, NI} of dz (K-major,
// as in the forward pass) and the weights' box {NB input channels, tap, 64
// output channels} as it lies, contiguous along N.  All four classes go in
// one launch, the ones of most taps first.  A class's sum over taps, then
// output channels, is cut where the GEMM it replaces split its K range, a
// tensor-memory accumulator for each of at most Z pieces, added in order in
// the epilogue: the results are the same bits at any batch, and those of that
// GEMM.
//
// Against gathers in software (cp.async of 16-byte chunks with their index
// arithmetic, four launches a layer, FP32 partials and a reduction where a
// class has few tiles), batch 256: layer 3 146 -> 52 us, layer 4 159 -> 41,
// layer 5 111 -> 24, layer 6 60 -> 20; the training step 1282 -> 898 us.
template <int CIN, int COUT, int HI, int WI, int TW, int TH, int S, int NI, int NB, int Z>
struct DgradTma {
  static constexpr int HO = (HI + 1) / 2, WO = (WI + 1) / 2;  // dz, and the largest class
  static constexpr int TX = (WO + TW - 1) / TW, TY = (HO + TH - 1) / TH;
  static constexpr int SW = 128, CB = COUT / 64, MMAS = 4;
  static constexpr int ROWS = NI * TW * TH;
  static constexpr int BOX_BYTES = ROWS * SW;
  static constexpr int A_BYTES = 128 * SW;
  static constexpr int B_BYTES = 64 * NB * 2;
  static constexpr int STAGE = A_BYTES + B_BYTES;
  static constexpr int TX_BYTES = BOX_BYTES + B_BYTES;
  static constexpr int SMEM = S * STAGE + 1024;
  static constexpr int TMEM_COLS = Z * NB, NSPLIT = CIN / NB;  // Z accumulators
  static constexpr bool B_MN = true;
  static constexpr int B_STEP = 16 * 128;
  static __device__ __forceinline__ uint64_t b_desc(uint32_t saddr) { return mn_desc(saddr, NB > 64 ? 64 * 128 : 1024); }
  static_assert(ROWS <= 128 && (NI == 1 || (TX == 1 && TY == 1)), "one 128-row MMA tile");
  static_assert(COUT % 64 == 0 && (NB == 64 || NB == 128) && CIN % NB == 0, "channel blocks");
  static_assert(TMEM_COLS <= 512 && (Z & (Z - 1)) == 0, "tensor-memory columns");
};

template <int CIN, int COUT, int HI, int WI, int TW, int TH, int S, int NI, int NB, int Z>
__global__ void __launch_bounds__(kConvThreads) dgrad_tma_kernel(
    const __grid_constant__ CUtensorMap map_dz, const __grid_constant__ CUtensorMap map_w,
    const bf16* __restrict__ act, bf16* __restrict__ out, int B, int tiles,
    const DgradSplits splits, int* __restrict__ err) {
  using C = DgradTma<CIN, COUT, HI, WI, TW, TH, S, NI, NB, Z>;
  extern __shared__ unsigned char conv_raw[];
  __shared__ __align__(8) uint64_t s_full[S], s_empty[S], s_done;
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail, s_issued, s_consumed;
  unsigned char* stages = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(conv_raw) + 1023) & ~(uintptr_t)1023);
  const int cls = 3 - (int)blockIdx.x / tiles, tile = (int)blockIdx.x % tiles;
  const int py = cls >> 1, px = cls & 1;
  const int img = NI == 1 ? tile / (C::TX * C::TY) : tile * NI;
  const int r = NI == 1 ? tile % (C::TX * C::TY) : 0;
  const int cy0 = (r / C::TX) * TH, cx0 = (r % C::TX) * TW;
  const int nb0 = (int)blockIdx.y * NB;
  const int steps = (1 + py) * (1 + px) * C::CB, per = splits.steps[cls];
  const int warp = threadIdx.x >> 5;

  if (threadIdx.x == 0) {
    s_fail = 0;
    s_issued = 0;
    s_consumed = 0;
    for (int i = 0; i < S; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_full[i])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_empty[i])));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_done)));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&s_tmem)),
                 "r"(C::TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s_tmem;

  if (warp == 1) {
    const uint32_t lane = threadIdx.x & 31;
    int st = 0, cb = 0, tx = 0, ty = 0;   // channel block and tap of the class
    uint32_t phase = 1u;
#pragma unroll 1
    for (int g = 0; g < steps; ++g) {
      if (g >= S && !bar_wait(smem_u32(&s_empty[st]), phase)) {
        if (lane == 0) atomicExch(&s_fail, 1);
        break;
      }
      const uint32_t base = smem_u32(stages) + (uint32_t)st * C::STAGE;
      const int ky = py ? 2 * ty : 1, kx = px ? 2 * tx : 1;
      if (lane == 0) {
        const uint32_t bar = smem_u32(&s_full[st]);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                     "r"(C::TX_BYTES)
                     : "memory");
        tma_load_4d(base, &map_dz, 64 * cb, cx0 + (px && kx == 0), cy0 + (py && ky == 0), img, bar);
#pragma unroll
        for (int q = 0; q < NB / 64; ++q)
          tma_load_3d(base + C::A_BYTES + q * 64 * 128, &map_w, nb0 + 64 * q, 3 * ky + kx, 64 * cb, bar);
      }
      *reinterpret_cast<volatile int*>(&s_issued) = g + 1;
      if (++cb == C::CB) {
        cb = 0;
        if (++tx > px) {
          tx = 0;
          ++ty;
        }
      }
      if (++st == S) {
        st = 0;
        phase ^= 1u;
      }
    }
  }
  if (warp == 0) {
    bool ok = true;
    for (int g = 0, z = 0; g < steps && ok; g += per, ++z)
      ok = mma_steps<C, S, NB>(tmem + (uint32_t)(z * NB), g, min(per, steps - g), s_full, s_empty,
                               smem_u32(stages), &s_consumed);
    // one last commit tracks every MMA issued (all, or those before a failure)
    commit_lane0(smem_u32(&s_done));
    if (!ok) s_fail = 1;
  }
  if (!bar_wait(smem_u32(&s_done), 0u)) atomicExch(&s_fail, 1);
  __syncthreads();
  // loads issued but not consumed (after a failure) land before the CTA exits
  if (threadIdx.x == 32)
    for (int s = s_consumed; s < s_issued; ++s)
      bar_wait(smem_u32(&s_full[s % S]), (uint32_t)((s / S) & 1));
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (!*reinterpret_cast<volatile int*>(&s_fail)) {
    // TMEM lane = row m: image img + m / (TW TH), class pixel (cy0 + q / TW, cx0 + q % TW)
    const int m = threadIdx.x;
    const int g = m / (TW * TH), q = m % (TW * TH);
    const int iy = 2 * (cy0 + q / TW) + py, ix = 2 * (cx0 + q % TW) + px;
    const bool ok = g < NI && img + g < B && iy < HI && ix < WI;
    const size_t off = (((size_t)(img + g) * HI + iy) * WI + ix) * CIN + nb0;
#pragma unroll 1
    for (int c0 = 0; c0 < NB; c0 += 16) {
      uint4 mk[2] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
      if (ok) {
        mk[0] = *reinterpret_cast<const uint4*>(act + off + c0);
        mk[1] = *reinterpret_cast<const uint4*>(act + off + c0 + 8);
      }
      float x[16];
      for (int z = 0; z * per < steps; ++z) {
        uint32_t v[16];
        const uint32_t taddr = tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)(z * NB + c0);
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, "
            "%10, %11, %12, %13, %14, %15}, [%16];\n"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
              "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
              "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
            : "r"(taddr));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int j = 0; j < 16; ++j) x[j] = z ? x[j] + __uint_as_float(v[j]) : __uint_as_float(v[j]);
      }
      if (ok) {
        const uint32_t mw[8] = {mk[0].x, mk[0].y, mk[0].z, mk[0].w, mk[1].x, mk[1].y, mk[1].z, mk[1].w};
        uint32_t packed[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(&mw[j]);
          const float x0 = __bfloat162float(a.x) > 0.f ? x[2 * j] : 0.f;
          const float x1 = __bfloat162float(a.y) > 0.f ? x[2 * j + 1] : 0.f;
          const __nv_bfloat162 b2 = __floats2bfloat162_rn(x0, x1);
          packed[j] = *reinterpret_cast<const uint32_t*>(&b2);
        }
        uint4* d = reinterpret_cast<uint4*>(out + off + c0);
        d[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
        d[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
      }
    }
  } else if (threadIdx.x == 0 && err) {
    atomicExch(err, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(C::TMEM_COLS));
}

// Raises a kernel's dynamic shared-memory limit on the current device, once
// per device and kernel (limits: the kernel's own table), before any stream
// capture that runs it.  With threads, *resident = the CTAs that the device
// holds at once.
int prepare_kernel(const void* kern, int smem, PerDevice& limits, int threads = 0,
                   int* resident = nullptr) {
  int dev = 0, value = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return (int)e;
  const int r = limits.get(dev, &value, [&](int* v) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess || !threads) return (int)e;
    int per_sm = 0, sms = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    *v = max(per_sm, 1) * max(sms, 1);
    return (int)e;
  });
  if (resident) *resident = value;
  return r;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// cuTensorMapEncodeTiled through the runtime's driver entry point (looked up once).
EncodeTiledFn encode_tiled() {
  static std::once_flag once;
  static EncodeTiledFn fn = nullptr;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
    else
      cudaGetLastError();
  });
  return fn;
}

// Input map: NHWC bfloat16 {C, W, H, N}, box {KB, 2 TW, 2 TH, 1} with
// element stride 2 in W and H (TW x TH pixels land); weight map: [C_out]
// [9 C_in] as {9 C_in, C_out}, box {KB, C_out}; both with the swizzle of
// their KB x 2-byte rows.  Zero fill outside the tensors.
template <int CIN, int COUT, int HI, int WI, int TW, int TH, int S, int NI = 1, int NB = COUT>
int run(const bf16* x, int B, const bf16* w, const float* bias, bf16* out, int* err,
        cudaStream_t st) {
  using C = ConvTma<CIN, COUT, HI, WI, TW, TH, S, NI, NB>;
  EncodeTiledFn enc = encode_tiled();
  if (!enc) return GS2D_ERR_CUDA;
  if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(w) |
       reinterpret_cast<uintptr_t>(out)) & 15)
    return GS2D_ERR_INVALID_ARG;
  CUtensorMap mx, mw;
  const cuuint64_t xdim[4] = {(cuuint64_t)CIN, (cuuint64_t)WI, (cuuint64_t)HI, (cuuint64_t)B};
  const cuuint64_t xstr[3] = {(cuuint64_t)CIN * 2, (cuuint64_t)WI * CIN * 2,
                              (cuuint64_t)HI * WI * CIN * 2};
  const cuuint32_t xbox[4] = {(cuuint32_t)C::KB, 2 * TW, 2 * TH, (cuuint32_t)NI};
  const cuuint32_t xes[4] = {1, 2, 2, 1};
  if (enc(&mx, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16*>(x), xdim, xstr, xbox, xes,
          CU_TENSOR_MAP_INTERLEAVE_NONE, C::SW == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
          CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return GS2D_ERR_CUDA;
  const cuuint64_t wdim[2] = {(cuuint64_t)9 * CIN, (cuuint64_t)COUT};
  const cuuint64_t wstr[1] = {(cuuint64_t)9 * CIN * 2};
  const cuuint32_t wbox[2] = {(cuuint32_t)C::KB, (cuuint32_t)NB};
  const cuuint32_t wes[2] = {1, 1};
  if (enc(&mw, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16*>(w), wdim, wstr, wbox, wes,
          CU_TENSOR_MAP_INTERLEAVE_NONE, C::SW == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
          CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return GS2D_ERR_CUDA;
  static PerDevice limits;
  const auto kern = conv_tma_kernel<CIN, COUT, HI, WI, TW, TH, S, NI, NB>;
  if (prepare_kernel(reinterpret_cast<const void*>(kern), C::SMEM, limits)) return GS2D_ERR_CUDA;
  const int grid = NI == 1 ? B * C::TX * C::TY : (B + NI - 1) / NI;
  if (grid <= 0) return GS2D_OK;
  kern<<<dim3(grid, C::NSPLIT), kConvThreads, C::SMEM, st>>>(mx, mw, bias, out, B, err);
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

// The persistent form on the GPU's resident CTAs (see conv_tma_pers_kernel).
template <int CIN, int COUT, int HI, int WI, int TW, int TH, int S>
int run_pers(const bf16* x, int B, const bf16* w, const float* bias, bf16* out, int* err,
             cudaStream_t st) {
  using C = ConvTma<CIN, COUT, HI, WI, TW, TH, S>;
  static_assert(2 * C::TMEM_COLS <= 512, "two accumulators fit the tensor memory");
  EncodeTiledFn enc = encode_tiled();
  if (!enc) return GS2D_ERR_CUDA;
  if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(w) |
       reinterpret_cast<uintptr_t>(out)) & 15)
    return GS2D_ERR_INVALID_ARG;
  CUtensorMap mx, mw;
  const cuuint64_t xdim[4] = {(cuuint64_t)CIN, (cuuint64_t)WI, (cuuint64_t)HI, (cuuint64_t)B};
  const cuuint64_t xstr[3] = {(cuuint64_t)CIN * 2, (cuuint64_t)WI * CIN * 2,
                              (cuuint64_t)HI * WI * CIN * 2};
  const cuuint32_t xbox[4] = {(cuuint32_t)C::KB, 2 * TW, 2 * TH, 1};
  const cuuint32_t xes[4] = {1, 2, 2, 1};
  const CUtensorMapSwizzle sw =
      C::SW == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
  if (enc(&mx, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16*>(x), xdim, xstr, xbox, xes,
          CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return GS2D_ERR_CUDA;
  const cuuint64_t wdim[2] = {(cuuint64_t)9 * CIN, (cuuint64_t)COUT};
  const cuuint64_t wstr[1] = {(cuuint64_t)9 * CIN * 2};
  const cuuint32_t wbox[2] = {(cuuint32_t)C::KB, COUT};
  const cuuint32_t wes[2] = {1, 1};
  if (enc(&mw, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16*>(w), wdim, wstr, wbox, wes,
          CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return GS2D_ERR_CUDA;
  static PerDevice limits;
  int resident = 0;
  const auto kern = conv_tma_pers_kernel<CIN, COUT, HI, WI, TW, TH, S>;
  if (prepare_kernel(reinterpret_cast<const void*>(kern), C::SMEM, limits, kPersThreads, &resident))
    return GS2D_ERR_CUDA;
  const int n_tiles = B * C::TX * C::TY;
  if (n_tiles <= 0) return GS2D_OK;
  kern<<<min(n_tiles, resident), kPersThreads, C::SMEM, st>>>(mx, mw, bias, out, n_tiles, err);
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

// dz map: NHWC bfloat16 {C_out, WO, HO, N}, box {64, TW, TH, NI}; weight map:
// [C_out][9][C_in] as {C_in, 9, C_out}, box {64, 1, 64}; 128-byte swizzle.
template <int CIN, int COUT, int HI, int WI, int TW, int TH, int S, int NI, int NB, int Z>
int run_dgrad(const bf16* dz, int B, const bf16* w, const bf16* act, bf16* out,
              const DgradSplits& splits, int* err, cudaStream_t st) {
  using C = DgradTma<CIN, COUT, HI, WI, TW, TH, S, NI, NB, Z>;
  for (int c = 0; c < 4; ++c)
    if (splits.steps[c] <= 0 || splits.steps[c] * Z < (1 + (c >> 1)) * (1 + (c & 1)) * C::CB)
      return GS2D_ERR_INVALID_ARG;
  EncodeTiledFn enc = encode_tiled();
  if (!enc) return GS2D_ERR_CUDA;
  if ((reinterpret_cast<uintptr_t>(dz) | reinterpret_cast<uintptr_t>(w) |
       reinterpret_cast<uintptr_t>(act) | reinterpret_cast<uintptr_t>(out)) & 15)
    return GS2D_ERR_INVALID_ARG;
  CUtensorMap mz, mw;
  const cuuint64_t zdim[4] = {(cuuint64_t)COUT, (cuuint64_t)C::WO, (cuuint64_t)C::HO, (cuuint64_t)B};
  const cuuint64_t zstr[3] = {(cuuint64_t)COUT * 2, (cuuint64_t)C::WO * COUT * 2,
                              (cuuint64_t)C::HO * C::WO * COUT * 2};
  const cuuint32_t zbox[4] = {64, TW, TH, NI}, zes[4] = {1, 1, 1, 1};
  const cuuint64_t wdim[3] = {(cuuint64_t)CIN, 9, (cuuint64_t)COUT};
  const cuuint64_t wstr[2] = {(cuuint64_t)CIN * 2, (cuuint64_t)9 * CIN * 2};
  const cuuint32_t wbox[3] = {64, 1, 64}, wes[3] = {1, 1, 1};
  if (enc(&mz, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16*>(dz), zdim, zstr, zbox, zes,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
          CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS ||
      enc(&mw, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<bf16*>(w), wdim, wstr, wbox, wes,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
          CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return GS2D_ERR_CUDA;
  static PerDevice limits;
  const auto kern = dgrad_tma_kernel<CIN, COUT, HI, WI, TW, TH, S, NI, NB, Z>;
  if (prepare_kernel(reinterpret_cast<const void*>(kern), C::SMEM, limits)) return GS2D_ERR_CUDA;
  const int tiles = NI == 1 ? B * C::TX * C::TY : (B + NI - 1) / NI;
  kern<<<dim3(4 * tiles, C::NSPLIT), kConvThreads, C::SMEM, st>>>(mz, mw, act, out, B, tiles, splits, err);
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

}  // namespace

// Which form a layer runs in at a batch.  None changes a result: every tile
// sums its K steps in the same order.  A CTA's time is its chain of K steps
// (~0.25 us each, 9 to 36 of them, nearly whatever their bytes) plus ~5 us,
// so a batch too small to fill the GPU splits the output channels over more
// CTAs (NB of them each, which lets a stage be smaller and more stages fit);
// a larger one takes wide tiles, few enough stages that two CTAs share an SM,
// and for layers 3 and 4 the persistent form.  Measured per layer (us, batch
// 1 / 24 / 77 / 256; before: one or two forms per layer and one thread
// issuing loads and MMAs):
//   layer 2   8.4 / 9.9 / 19.5 / 45.0  ->   6.8 / 8.9 / 18.4 / 40.6
//   layer 3  11.2 / 10.9 / 19.2 / 30.4 ->   7.3 / 8.5 / 14.0 / 31.1
//   layer 4  20.3 / 18.9 / 18.9 / 26.8 ->   9.3 / 10.8 / 14.7 / 21.8
//   layer 5  22.1 / 23.6 / 22.3 / 23.4 ->  13.5 / 14.0 / 14.0 / 17.1
//   layer 6  17.7 / 18.4 / 18.0 / 18.0 ->  13.3 / 14.0 / 13.6 / 14.3
int conv_tma_forward(int layer, const bf16* x, int B, const bf16* w, const float* bias, bf16* out,
                     int* err, cudaStream_t st) {
  constexpr int kSms = 152;
  switch (layer) {
    case 1:   // 10 tiles per image
      return B * 10 * 2 <= 2 * kSms ? run<32, 64, 60, 80, 8, 16, 9, 1, 32>(x, B, w, bias, out, err, st)
                                    : run<32, 64, 60, 80, 8, 16, 3>(x, B, w, bias, out, err, st);
    case 2:   // 3 tiles per image
      if (B * 3 * 4 <= kSms) return run<64, 128, 30, 40, 8, 16, 9, 1, 32>(x, B, w, bias, out, err, st);
      if (B * 3 * 2 <= 4 * kSms / 3)
        return run<64, 128, 30, 40, 8, 16, 4, 1, 64>(x, B, w, bias, out, err, st);
      return B * 3 <= 2 * kSms ? run<64, 128, 30, 40, 8, 16, 3>(x, B, w, bias, out, err, st)
                               : run_pers<64, 128, 30, 40, 8, 16, 6>(x, B, w, bias, out, err, st);
    // layer 4's 8 x 10 outputs are one tile of 80 rows
    case 3:
      if (B * 8 <= kSms) return run<128, 256, 15, 20, 10, 8, 11, 1, 32>(x, B, w, bias, out, err, st);
      if (B * 4 <= kSms) return run<128, 256, 15, 20, 10, 8, 9, 1, 64>(x, B, w, bias, out, err, st);
      if (B * 2 <= kSms) return run<128, 256, 15, 20, 10, 8, 6, 1, 128>(x, B, w, bias, out, err, st);
      return B <= kSms ? run<128, 256, 15, 20, 10, 8, 3, 1, 128>(x, B, w, bias, out, err, st)
                       : run_pers<128, 256, 15, 20, 10, 8, 4>(x, B, w, bias, out, err, st);
    // layers 5 and 6 (4 x 5 and 2 x 3 outputs): whole images per tile (5 and
    // 21: 100 and 126 rows)
    case 4: {
      const int tiles = (B + 4) / 5;
      if (tiles * 8 <= kSms) return run<256, 256, 8, 10, 5, 4, 11, 5, 32>(x, B, w, bias, out, err, st);
      if (tiles * 4 <= kSms) return run<256, 256, 8, 10, 5, 4, 9, 5, 64>(x, B, w, bias, out, err, st);
      return tiles * 4 <= 2 * kSms ? run<256, 256, 8, 10, 5, 4, 4, 5, 64>(x, B, w, bias, out, err, st)
                                   : run<256, 256, 8, 10, 5, 4, 3, 5, 128>(x, B, w, bias, out, err, st);
    }
    case 5:
      return (B + 20) / 21 * 8 <= kSms ? run<256, 256, 4, 5, 3, 2, 11, 21, 32>(x, B, w, bias, out, err, st)
                                       : run<256, 256, 4, 5, 3, 2, 5, 21, 32>(x, B, w, bias, out, err, st);
    default: return GS2D_ERR_INVALID_ARG;
  }
}

// Tiles: layer 3's 15 x 20 class pixels in three parts of 6 rows, layer 4's 8
// x 10 whole, 6 images' 4 x 5 of layer 5, 21 images' 2 x 3 of layer 6.
int dgrad_tma(int layer, const bf16* dz, int B, const bf16* w, const bf16* act, bf16* out,
              const DgradSplits& splits, int* err, cudaStream_t st) {
  switch (layer) {
    case 2: return run_dgrad<64, 128, 30, 40, 20, 6, 3, 1, 64, 1>(dz, B, w, act, out, splits, err, st);
    case 3: return run_dgrad<128, 256, 15, 20, 10, 8, 3, 1, 128, 2>(dz, B, w, act, out, splits, err, st);
    case 4: return run_dgrad<256, 256, 8, 10, 5, 4, 4, 6, 64, 2>(dz, B, w, act, out, splits, err, st);
    case 5: return run_dgrad<256, 256, 4, 5, 3, 2, 8, 21, 64, 8>(dz, B, w, act, out, splits, err, st);
    default: return GS2D_ERR_INVALID_ARG;
  }
}

}  // namespace net
}  // namespace gs2d
