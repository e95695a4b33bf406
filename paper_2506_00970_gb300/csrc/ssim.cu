// SSIM term of the mapping loss (Sec. III-E, L_c with L_SSIM; SSIM of Wang
// et al. 2004 with the 11 x 11 Gaussian window, sigma 1.5, C1 = 0.01^2,
// C2 = 0.03^2 for images in [0, 1]) and its gradient, in one fused pass.
//
// Per channel and pixel p, with the window w (zero padding at the border),
// the usual statistics mu_x = w * x, mu_y, sigma_x^2 = w * x^2 - mu_x^2,
// sigma_y^2, sigma_xy give
//   S = (2 mu_x mu_y + C1)(2 sigma_xy + C2) /
//       ((mu_x^2 + mu_y^2 + C1)(sigma_x^2 + sigma_y^2 + C2)).
// FP32 loses that form to cancellation where x ~ y (the numerator and the
// denominator agree to many digits, and so do the terms of its gradient),
// so the kernel works with the difference image d = x - y: with
// mu_d = w * d and sigma_d^2 = w * d^2 - mu_d^2 (identities:
// 2 mu_x mu_y + C1 = b1 - mu_d^2, 2 sigma_xy + C2 = b2 - sigma_d^2),
//   S = (1 - mu_d^2 / b1)(1 - sigma_d^2 / b2),
//   b1 = mu_x^2 + mu_y^2 + C1,  b2 = sigma_x^2 + sigma_y^2 + C2,
// so 1 - S = p + q - p q with p = mu_d^2 / b1, q = sigma_d^2 / b2 and the
// partial derivatives w.r.t. the moments (mu_x, mu_d, E_xx, E_yy, E_dd)
// have no large cancelling terms.  The loss adds
// weight / |Omega| sum_p (1 - mean_c S_c(p)); with G_* the partials of S
// times the upstream -weight / (3 |Omega|), the gradient w.r.t. x is
//   w * (G_mux + G_mud) + 2 x (w * G_xx) + 2 d (w * G_dd)
// (the window is symmetric, so the adjoint filter is the same filter).
//
// One block per 32 x 32 output tile and channel.  It stages x and y on the
// tile plus a 10-pixel ring in shared memory and filters the five moment maps
// separably on the tile plus a 5-pixel ring (columns, then rows), evaluates
// S and the three G maps there (zero outside the image), filters those
// separably down to the tile (rows, then columns) and writes the gradient.
// Everything between the image reads and the gradient write stays in shared
// memory: per pixel and channel the kernel reads x and y and adds one
// gradient value.  The per-block loss sums are reduced in a fixed order
// (deterministic).
//
// The kernel is bound by its FP32 issue, so every filter runs on pairs
// (fma.rn.f32x2, two values per instruction): a column filter takes adjacent
// columns, which lie side by side in a row-major map; its results are stored
// transposed, so that the row filter that follows finds adjacent rows side by
// side.  A thread forms four outputs along the filter from one pass over
// their fourteen taps, and the products x^2, y^2, d^2 once per tap instead of
// once per tap and output.  Six outputs per thread in 192 threads left too
// few warps to cover the phases' barriers.  1200x680, three channels: 81 us
// with one value per instruction, 72 us with pairs in 192 threads, 68 us
// so.
#include <cmath>

#include "f32x2.cuh"
#include "gs2d_common.cuh"
#include "gs2d_internal.h"
#include "per_device.h"

namespace gs2d {

constexpr int kSsimT = 32;                 // output tile edge
constexpr int kSsimR = 5;                  // window radius
constexpr int kSsimA = kSsimT + 4 * kSsimR;  // 52: staged edge (two rings)
constexpr int kSsimB = kSsimT + 2 * kSsimR;  // 42: moment / G map edge
constexpr int kSsimThreads = 288;
constexpr float kSsimC1 = 0.0001f, kSsimC2 = 0.0009f;
constexpr float kSsimTame = 4.f;

struct SsimWin {
  float g[2 * kSsimR + 1];  // normalised 1D Gaussian; the window is g g^T
};

// Shared memory (floats).  Region A: x and y (2 x 52 rows of 52), later the
// three G maps, transposed (3 x 42 columns of 46 rows).  Region B: the five
// column-filtered moment maps, transposed (5 x 52 columns of 46 rows), later
// the three row-filtered G maps (3 x 42 rows of 36).  Pitches are even (pairs
// of floats are read) and spread a warp's stores over the banks (two-way
// conflicts at most).
constexpr int kSsimBP = 46;                       // pitch of the 42-row transposed maps
constexpr int kSsimFP = 36;                       // pitch of the 32-column filtered G maps
constexpr int kSsimSmemA = 3 * kSsimB * kSsimBP;
// two columns of slack: the last group of a filter reads past the 52 columns
// (rows) for outputs beyond the 42, which are dropped
constexpr int kSsimSmemB = (5 * kSsimA + 2) * kSsimBP;
constexpr size_t kSsimSmemBytes = (size_t)(kSsimSmemA + kSsimSmemB) * sizeof(float);
static_assert((2 * kSsimA + 2) * kSsimA <= kSsimSmemA, "x, y and two rows of slack fit region A");
static_assert(3 * kSsimB * kSsimFP <= kSsimSmemB, "filtered G maps fit region B");
static_assert(kSsimSmemA % 4 == 0 && kSsimFP % 4 == 0, "16-byte stores");
constexpr int kSsimM = 4;                         // outputs per thread of a filter
constexpr int kSsimGM = (kSsimB + kSsimM - 1) / kSsimM;   // 11 groups of the moment filters
constexpr int kSsimGG = kSsimT / kSsimM;                  // 8 groups of the G row filter
constexpr int kSsimC = 2;                         // outputs per thread of the last filter
constexpr int kSsimTaps = 2 * kSsimR + 1;

// acc[o] += sum over taps t of w_t v[o + t], fed one value at a time: i is
// the index of v (taps i - o of the outputs it reaches).
template <int kOut, int kMaps>
__device__ __forceinline__ void filter_tap(const F2 (&w)[kSsimR + 1], const F2 (&v)[kMaps], int i,
                                           F2 (&acc)[kMaps][kOut]) {
#pragma unroll
  for (int o = 0; o < kOut; ++o) {
    const int t = i - o;
    if (t < 0 || t >= kSsimTaps) continue;
    const F2 g = w[t <= kSsimR ? t : 2 * kSsimR - t];
#pragma unroll
    for (int k = 0; k < kMaps; ++k) acc[k][o] = fma2(g, v[k], acc[k][o]);
  }
}

__global__ void __launch_bounds__(kSsimThreads, 3) ssim_kernel(const float* __restrict__ x,
                                                           const float* __restrict__ y, int H,
                                                           int W, float weight, SsimWin win,
                                                           float* __restrict__ g_x,
                                                           float* __restrict__ part) {
  extern __shared__ float4 smem4[];
  float* sa = reinterpret_cast<float*>(smem4);    // x, y [52][52]  ->  G [3][42 q][46 r]
  float* sb = sa + kSsimSmemA;                    // M [5][52 q][46 r]  ->  F [3][42 r][36 q]
  __shared__ float s_red[kSsimThreads / 32];
  const int c = blockIdx.z;
  const int tx0 = blockIdx.x * kSsimT, ty0 = blockIdx.y * kSsimT;
  const int ax0 = tx0 - 2 * kSsimR, ay0 = ty0 - 2 * kSsimR;   // staged origin
  F2 w[kSsimR + 1];
#pragma unroll
  for (int t = 0; t <= kSsimR; ++t) w[t] = dup2(win.g[t]);
  // stage x, y (zero outside the image), a warp per row: the lanes' columns
  // and offsets are the same in every row.  Where no value exceeds kSsimTame,
  // b1 and b2 are in [C2 / 2, 100] despite the rounding of their differences
  // (4e-6 of 16 each), and recip2 need not divide
  bool tame = true;
  {
    constexpr int kW = kSsimThreads / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int qa = lane, qb = lane + 32;
    const bool ia = ax0 + qa >= 0 && ax0 + qa < W;
    const bool ib = qb < kSsimA && ax0 + qb >= 0 && ax0 + qb < W;
    const float* px = x + ((ptrdiff_t)ay0 * W + ax0 + qa) * 3 + c;
    const float* py = y + ((ptrdiff_t)ay0 * W + ax0 + qa) * 3 + c;
#pragma unroll 3
    for (int r = warp; r < kSsimA; r += kW) {
      const bool in = ay0 + r >= 0 && ay0 + r < H;
      const ptrdiff_t o = (ptrdiff_t)r * W * 3;
      const float xa = in && ia ? __ldg(px + o) : 0.f, ya = in && ia ? __ldg(py + o) : 0.f;
      const float xb = in && ib ? __ldg(px + o + 96) : 0.f, yb = in && ib ? __ldg(py + o + 96) : 0.f;
      tame = tame && fmaxf(fabsf(xa), fabsf(ya)) <= kSsimTame && fmaxf(fabsf(xb), fabsf(yb)) <= kSsimTame;
      float* d = sa + r * kSsimA + qa;
      d[0] = xa;
      d[kSsimA * kSsimA] = ya;
      if (qb < kSsimA) {
        d[32] = xb;
        d[kSsimA * kSsimA + 32] = yb;
      }
    }
  }
  tame = __syncthreads_and(tame) != 0;
  // column filter of the five moments (x, d = x - y, x^2, y^2, d^2) of the
  // columns 2 p, 2 p + 1: M[k][q][r0 .. r0 + 3] (rows 42, 43 land in the padding)
  for (int e = threadIdx.x; e < (kSsimA / 2) * kSsimGM; e += kSsimThreads) {
    const int p = e % (kSsimA / 2), r0 = (e / (kSsimA / 2)) * kSsimM;
    const float* sx = sa + r0 * kSsimA + 2 * p;
    const float* sy = sx + kSsimA * kSsimA;
    F2 acc[5][kSsimM];
#pragma unroll
    for (int k = 0; k < 5; ++k)
#pragma unroll
      for (int o = 0; o < kSsimM; ++o) acc[k][o] = dup2(0.f);
#pragma unroll
    for (int i = 0; i < kSsimM + 2 * kSsimR; ++i) {
      const F2 a = load2(sx + i * kSsimA), b = load2(sy + i * kSsimA);
      const F2 d = sub2(a, b);
      const F2 v[5] = {a, d, mul2(a, a), mul2(b, b), mul2(d, d)};
      filter_tap(w, v, i, acc);
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      float* col = sb + (k * kSsimA + 2 * p) * kSsimBP + r0;
#pragma unroll
      for (int o = 0; o < kSsimM; o += 2) {
        const float2 u = split2(acc[k][o]), v = split2(acc[k][o + 1]);
        *reinterpret_cast<float2*>(col + o) = make_float2(u.x, v.x);
        *reinterpret_cast<float2*>(col + kSsimBP + o) = make_float2(u.y, v.y);
      }
    }
  }
  __syncthreads();
  // row filter of the rows 2 p, 2 p + 1, then S and the G maps at their
  // columns q0 .. q0 + 3 of the 42 x 42 region (origin tile - 5); x and y are
  // dead, so the G maps take region A
  const float up = -weight / (3.f * (float)H * (float)W);
  float loss = 0.f;
  for (int e = threadIdx.x; e < (kSsimB / 2) * kSsimGM; e += kSsimThreads) {
    const int p = e % (kSsimB / 2), q0 = (e / (kSsimB / 2)) * kSsimM;
    F2 acc[5][kSsimM];
#pragma unroll
    for (int k = 0; k < 5; ++k)
#pragma unroll
      for (int o = 0; o < kSsimM; ++o) acc[k][o] = dup2(0.f);
#pragma unroll
    for (int i = 0; i < kSsimM + 2 * kSsimR; ++i) {
      F2 v[5];
#pragma unroll
      for (int k = 0; k < 5; ++k) v[k] = load2(sb + (k * kSsimA + q0 + i) * kSsimBP + 2 * p);
      filter_tap(w, v, i, acc);
    }
    // the reciprocals of the four outputs' denominators, with one branch for all:
    // a division, or a branch around it, in each output keeps the outputs from
    // overlapping (whole SSIM pass at 1200x680: 66.5 us with approximations
    // only, 2 us more so, 67.6 with the one branch)
    F2 ib[kSsimM][2];
#pragma unroll
    for (int o = 0; o < kSsimM; ++o) {
      const F2 mx = acc[0][o], my = sub2(mx, acc[1][o]);
      ib[o][0] = fma2(mx, mx, fma2(my, my, dup2(kSsimC1)));
      ib[o][1] = add2(add2(sub2(acc[2][o], mul2(mx, mx)), sub2(acc[3][o], mul2(my, my))),
                      dup2(kSsimC2));
    }
    if (tame) {
#pragma unroll
      for (int o = 0; o < kSsimM; ++o) {
        ib[o][0] = recip2<true>(ib[o][0]);
        ib[o][1] = recip2<true>(ib[o][1]);
      }
    } else {
#pragma unroll
      for (int o = 0; o < kSsimM; ++o) {
        ib[o][0] = recip2<false>(ib[o][0]);
        ib[o][1] = recip2<false>(ib[o][1]);
      }
    }
#pragma unroll
    for (int o = 0; o < kSsimM; ++o) {
      const int q = q0 + o, px = tx0 - kSsimR + q, py = ty0 - kSsimR + 2 * p;
      if (q >= kSsimB) break;
      const F2 mx = acc[0][o], md = acc[1][o], my = sub2(mx, md);
      const F2 one = dup2(1.f);
      const F2 vd = sub2(acc[4][o], mul2(md, md));
      const F2 ib1 = ib[o][0], ib2 = ib[o][1];
      const F2 p1 = mul2(mul2(md, md), ib1), q1 = mul2(vd, ib2);   // 1 - P, 1 - Q
      const F2 P = sub2(one, p1), Q = sub2(one, q1);
      const F2 dmx = mul2(mul2(dup2(2.f), add2(mx, my)),
                          sub2(mul2(mul2(Q, p1), ib1), mul2(mul2(P, q1), ib2)));
      const F2 dmd = fma2(mul2(mul2(Q, dup2(-2.f)), ib1), fma2(my, p1, md),
                          mul2(mul2(mul2(P, dup2(2.f)), ib2), fma2(my, q1, md)));
      const F2 u2 = dup2(up), Pi = mul2(mul2(u2, P), ib2);
      const float2 g0 = split2(mul2(u2, add2(dmx, dmd))), g1 = split2(mul2(Pi, q1));
      const float2 g2 = split2(Pi), l = split2(sub2(add2(p1, q1), mul2(p1, q1)));   // 1 - S
      const bool in_x = px >= 0 && px < W;
      const bool i0 = in_x && py >= 0 && py < H, i1 = in_x && py + 1 >= 0 && py + 1 < H;
      if (q >= kSsimR && q < kSsimR + kSsimT) {
        if (i0 && 2 * p >= kSsimR && 2 * p < kSsimR + kSsimT) loss += l.x;
        if (i1 && 2 * p + 1 >= kSsimR && 2 * p + 1 < kSsimR + kSsimT) loss += l.y;
      }
      float* g = sa + q * kSsimBP + 2 * p;
      *reinterpret_cast<float2*>(g) = make_float2(i0 ? g0.x : 0.f, i1 ? g0.y : 0.f);
      *reinterpret_cast<float2*>(g + kSsimB * kSsimBP) =
          make_float2(i0 ? g1.x : 0.f, i1 ? g1.y : 0.f);
      *reinterpret_cast<float2*>(g + 2 * kSsimB * kSsimBP) =
          make_float2(i0 ? -g2.x : 0.f, i1 ? -g2.y : 0.f);
    }
  }
  if (g_x) {
    __syncthreads();
    // row filter of the G maps, a map per item, rows 2 p, 2 p + 1:
    // F[k][r][q0 .. q0 + 3]
    for (int e = threadIdx.x; e < 3 * (kSsimB / 2) * kSsimGG; e += kSsimThreads) {
      const int k = e / ((kSsimB / 2) * kSsimGG), j = e % ((kSsimB / 2) * kSsimGG);
      const int p = j % (kSsimB / 2), q0 = (j / (kSsimB / 2)) * kSsimM;
      F2 acc[1][kSsimM];
#pragma unroll
      for (int o = 0; o < kSsimM; ++o) acc[0][o] = dup2(0.f);
#pragma unroll
      for (int i = 0; i < kSsimM + 2 * kSsimR; ++i) {
        const F2 v[1] = {load2(sa + (k * kSsimB + q0 + i) * kSsimBP + 2 * p)};
        filter_tap(w, v, i, acc);
      }
      float2 u[kSsimM];
#pragma unroll
      for (int o = 0; o < kSsimM; ++o) u[o] = split2(acc[0][o]);
      float* row = sb + (k * kSsimB + 2 * p) * kSsimFP + q0;
      *reinterpret_cast<float4*>(row) = make_float4(u[0].x, u[1].x, u[2].x, u[3].x);
      *reinterpret_cast<float4*>(row + kSsimFP) = make_float4(u[0].y, u[1].y, u[2].y, u[3].y);
    }
    __syncthreads();
    // column filter to the tile (rows r0, r0 + 1 of columns 2 p, 2 p + 1) and
    // the gradient
    for (int e = threadIdx.x; e < (kSsimT / 2) * (kSsimT / kSsimC); e += kSsimThreads) {
      const int p = e % (kSsimT / 2), r0 = (e / (kSsimT / 2)) * kSsimC;
      const int px = tx0 + 2 * p;
      // the pixels' x, y and gradient so far, in flight during the filter
      float xv[kSsimC][2], yv[kSsimC][2], gv[kSsimC][2];
      bool in[kSsimC][2];
#pragma unroll
      for (int o = 0; o < kSsimC; ++o)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          in[o][h] = ty0 + r0 + o < H && px + h < W;
          const size_t i = ((size_t)(ty0 + r0 + o) * W + px + h) * 3 + c;
          xv[o][h] = in[o][h] ? __ldg(x + i) : 0.f;
          yv[o][h] = in[o][h] ? __ldg(y + i) : 0.f;
          gv[o][h] = in[o][h] ? g_x[i] : 0.f;
        }
      F2 acc[3][kSsimC];
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int o = 0; o < kSsimC; ++o) acc[k][o] = dup2(0.f);
#pragma unroll
      for (int i = 0; i < kSsimC + 2 * kSsimR; ++i) {
        F2 v[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) v[k] = load2(sb + (k * kSsimB + r0 + i) * kSsimFP + 2 * p);
        filter_tap(w, v, i, acc);
      }
#pragma unroll
      for (int o = 0; o < kSsimC; ++o) {
        const float2 f0 = split2(acc[0][o]), f1 = split2(acc[1][o]), f2 = split2(acc[2][o]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (!in[o][h]) continue;
          const size_t i = ((size_t)(ty0 + r0 + o) * W + px + h) * 3 + c;
          g_x[i] = gv[o][h] + fmaf(2.f * xv[o][h], h ? f1.y : f1.x,
                                   fmaf(2.f * (xv[o][h] - yv[o][h]), h ? f2.y : f2.x,
                                        h ? f0.y : f0.x));
        }
      }
    }
  }
  const float t = block_sum<kSsimThreads>(loss, s_red);
  if (threadIdx.x == 0)
    part[(blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = t;
}

// loss[0] += scale * (fixed-order sum of the block partials)
__global__ void ssim_sum_kernel(const float* __restrict__ part, int n, float scale,
                                float* __restrict__ loss) {
  __shared__ float s_red[8];
  float a = 0.f;
#pragma unroll 4
  for (int i = threadIdx.x; i < n; i += 256) a += part[i];
  const float t = block_sum256(a, s_red);
  if (threadIdx.x == 0) loss[0] += scale * t;
}

SsimWin ssim_window() {
  SsimWin w;
  double g[2 * kSsimR + 1], s = 0.0;
  for (int t = 0; t <= 2 * kSsimR; ++t) {
    const double d = t - kSsimR;
    g[t] = std::exp(-d * d / (2.0 * 1.5 * 1.5));
    s += g[t];
  }
  for (int t = 0; t <= 2 * kSsimR; ++t) w.g[t] = (float)(g[t] / s);
  return w;
}

size_t ssim_ws_bytes(int height, int width) {
  const size_t nb = (size_t)((width + kSsimT - 1) / kSsimT) * ((height + kSsimT - 1) / kSsimT) * 3;
  return align_up(nb * sizeof(float), 256);
}

int ssim_launch(const float* x, const float* y, int height, int width, float weight, float* g_x,
                float* loss, void* workspace, size_t ws_bytes, size_t* ws_needed,
                cudaStream_t st) {
  if (height <= 0 || width <= 0 || !x || !y || !loss) return GS2D_ERR_INVALID_ARG;
  const size_t need = ssim_ws_bytes(height, width);
  if (ws_needed) *ws_needed = need;
  if (!workspace || ws_bytes < need) return GS2D_ERR_WORKSPACE;
  static PerDevice limits;
  int dev = 0, unused = 0;
  GS2D_CUDA_TRY(cudaGetDevice(&dev));
  if (limits.get(dev, &unused, [](int*) {
        return (int)cudaFuncSetAttribute(ssim_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kSsimSmemBytes);
      }))
    return GS2D_ERR_CUDA;
  const dim3 grid((width + kSsimT - 1) / kSsimT, (height + kSsimT - 1) / kSsimT, 3);
  float* part = static_cast<float*>(workspace);
  ssim_kernel<<<grid, kSsimThreads, kSsimSmemBytes, st>>>(x, y, height, width, weight,
                                                          ssim_window(), g_x, part);
  GS2D_LAUNCH_CHECK();
  ssim_sum_kernel<<<1, 256, 0, st>>>(part, (int)(grid.x * grid.y * grid.z),
                                              weight / (3.f * (float)height * (float)width), loss);
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

}  // namespace gs2d

using namespace gs2d;

extern "C" {

size_t gs2d_ssim_workspace(int height, int width) { return ssim_ws_bytes(height, width); }

int gs2d_ssim_loss(const float* x, const float* y, int height, int width, float weight,
                   float* g_x, float* loss, void* workspace, size_t ws_bytes, size_t* ws_needed,
                   gs2d_stream stream) {
  return ssim_launch(x, y, height, width, weight, g_x, loss, workspace, ws_bytes, ws_needed,
                     (cudaStream_t)stream);
}

}  // extern "C"
