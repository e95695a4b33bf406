// Per-pixel loss kernels of tracking (Sec. III-D) and mapping (Sec. III-E):
// value and gradient w.r.t. the rendered images in one pass, per-block
// partial sums of the loss reduced in a fixed order.
#include "gs2d_common.cuh"
#include "gs2d_internal.h"
#include "loss_pixel.cuh"

namespace gs2d {

constexpr int kLossBlocks = 4 * 152;
constexpr int kLossThreads = 256;

// L_t = 1/|Omega| sum M_n M_o (|I_r - I|_1 + lambda_d |D_r - D|), Eq.
// tracking_loss; M_n = [N_r . r > 0] (Eq. normal_mask; r's length does not
// change the sign), M_o = [O > thresh] (Eq. opacity_mask); D_r = D/O in
// depth_mode 1.  Sub-gradient sign(0) = 0; the masks carry no gradient.
__global__ void __launch_bounds__(kLossThreads) tracking_loss_kernel(
    const float* __restrict__ rgb, const float* __restrict__ depth, const float* __restrict__ normal,
    const float* __restrict__ opac, const float* __restrict__ obs_rgb,
    const float* __restrict__ obs_depth, gs2d_camera cam, gs2d_track_params prm,
    float* __restrict__ g_rgb, float* __restrict__ g_depth, float* __restrict__ g_opac,
    float* __restrict__ part, const int32_t* __restrict__ gate) {
  __shared__ float s[kLossThreads / 32];
  if (gate && *gate) return;
  const int P = cam.width * cam.height;
  const float inv = 1.f / (float)P;
  float acc = 0.f;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P; i += gridDim.x * blockDim.x) {
    const float x = (i % cam.width) + 0.5f, y = (i / cam.width) + 0.5f;
    const float rx = (x - cam.cx) / cam.fx, ry = (y - cam.cy) / cam.fy;
    const PixLoss L = tracking_pixel_loss(
        f3(rgb[3 * i], rgb[3 * i + 1], rgb[3 * i + 2]), depth[i],
        f3(normal[3 * i], normal[3 * i + 1], normal[3 * i + 2]), opac[i],
        f3(obs_rgb[3 * i], obs_rgb[3 * i + 1], obs_rgb[3 * i + 2]), obs_depth[i], rx, ry, inv, prm);
    acc += L.loss;
    g_rgb[3 * i] = L.g_rgb[0];
    g_rgb[3 * i + 1] = L.g_rgb[1];
    g_rgb[3 * i + 2] = L.g_rgb[2];
    g_depth[i] = L.g_depth;
    g_opac[i] = L.g_opac;
  }
  const float t = block_sum256(acc, s);
  if (threadIdx.x == 0) part[blockIdx.x] = t * inv;
}

__global__ void __launch_bounds__(256) sum_parts_kernel(const float* __restrict__ part, int n,
                                                        float* __restrict__ out,
                                                        const int32_t* __restrict__ gate) {
  __shared__ float s[256];
  if (gate && *gate) return;
  float v = 0.f;
  for (int i = threadIdx.x; i < n; i += 256) v += part[i];
  s[threadIdx.x] = v;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h) s[threadIdx.x] += s[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = s[0];
}

// ---------------------------------------------------------------------------
// Mapping loss (Sec. III-E, colour term without SSIM):
//   per pixel |I_r - I|_1 + w_d |D_r/O - D| + w_n (1 - N_D . N_r),
// N_D = normalised cross product of the central differences of the
// back-projected points X = (D_r/O) r (Eq. normal_fromD), counted at interior
// pixels whose own and 4-neighbour opacities exceed 0.5.  The normal term's
// gradient w.r.t. the depth of pixel q collects the four stencils that use
// q, recomputed here (a gather, so no atomics).
//
// A warp takes a strip of 28 columns and R rows: a lane per column (two halo
// columns on each side) loads the depths and opacities of R + 4 rows at once
// and walks down them, keeping the normal term of the last two in registers;
// left and right neighbours come by shuffles.  Nothing is staged in shared
// memory and there is no block barrier.  Replaces 32 x 8 tiles with three
// barrier-separated phases over two rings in shared memory, which took ~650
// instructions a pixel (31 us at 1200x680, 197 us for eight such views, 7.9
// us at 160x120).  R = 4: 24, 140 and 11.8 us; taller strips repeat fewer
// halo rows but chain more latencies (R = 6: 21, 147, 14.5 us; R = 16: 45 us
// at 1200x680).
//
// Up to 200,000 pixels the strips are too few to hide those latencies among
// warps: R = 2, every input of the strip loaded before the first is used (with
// registers for 16 warps per SM, which is all there are), and in a batch
// blocks of two warps, so that they spread over the SMs.  Device time of a
// call in a graph, us, views of one size -- the tiles / R = 2 without that up to
// 136,000 pixels and R = 4 beyond / now:
//   1, 8 x 64x48     5.7  6.7  5.4     6.1  7.2  5.9
//   1, 8 x 160x120   6.6  7.1  5.8     8.7 10.5  8.0
//   1, 2 x 320x240   6.9  8.4  7.3     8.6 10.8  9.3
//   1, 2 x 480x360  10.6 11.4 10.1    15.5 12.9 13.0
//   one view's own call: 160x120  5.8 6.1 5.3, 320x240  7.3 7.0 6.4
constexpr int kStripW = 28;        // output columns of a strip
constexpr int kStripRows = 4;      // and rows
constexpr int kStripRowsSmall = 2;
constexpr int kSmallImages = 200000;   // pixels of a call
constexpr int kLossWarps = kLossThreads / 32;

__host__ __device__ inline int strips_along(int n, int step) { return (n + step - 1) / step; }
inline int strip_rows(long long px) { return px >= kSmallImages ? kStripRows : kStripRowsSmall; }
// Threads of a batch kernel's block, and blocks per SM of either kernel.
__host__ __device__ constexpr int batch_threads(int rows) {
  return rows == kStripRows ? kLossThreads : 64;
}
constexpr int loss_blocks_per_sm(int rows, int threads) {
  return (rows == kStripRows ? 32 : 16) / (threads / 32);
}

__device__ __forceinline__ F3 cross_rn(F3 a, F3 b) {
  return f3(fmaf(a.y, b.z, -__fmul_rn(a.z, b.y)), fmaf(a.z, b.x, -__fmul_rn(a.x, b.z)),
            fmaf(a.x, b.y, -__fmul_rn(a.y, b.x)));
}
__device__ __forceinline__ F3 fma_rn(float s, F3 a, F3 b) {
  return f3(fmaf(s, a.x, b.x), fmaf(s, a.y, b.y), fmaf(s, a.z, b.z));
}

struct MapLossImages {
  const float *rgb, *depth, *normal, *opac, *obs_rgb, *obs_depth;
  float *g_rgb, *g_depth, *g_normal, *g_opac;
};

// Gradients of the strip with first output pixel (x0, y0); returns the lane's
// sum of the loss terms (unscaled).  (ifx, ify) = (1/fx, 1/fy), taken once
// per kernel: the pixel ray is ((px + 0.5 - cx) ifx, (py + 0.5 - cy) ify, 1).
// Every product that is added to something is an explicit fmaf or __fmul_rn,
// so that the single-view and the batched kernel round alike and their
// gradients agree bit for bit, whatever the compiler would contract in each.
template <int R>
__device__ __forceinline__ float mapping_loss_strip(int x0, int y0,
                                                    const MapLossImages& im,
                                                    const gs2d_camera& cam, float ifx, float ify,
                                                    float inv, float w_l1, float w_d, float w_n) {
  const int W = cam.width, H = cam.height;
  const int lane = threadIdx.x & 31;
  const int px = x0 + lane - 2;
  const bool in_x = px >= 0 && px < W;
  const bool out_x = lane >= 2 && lane < 2 + kStripW && px < W;
  const float rxl = ((px - 1) + 0.5f - cam.cx) * ifx, rxc = (px + 0.5f - cam.cx) * ifx,
              rxr = ((px + 1) + 0.5f - cam.cx) * ifx;
  // D / max(O, 1e-6), O and D of rows y0 - 2 .. y0 + R + 1 (0 outside
  // the image)
  constexpr int kR = R + 4;
  constexpr bool kAhead = R == kStripRowsSmall;
  float dv[kR], ov[kR], Dv[kR];
#pragma unroll
  for (int k = 0; k < kR; ++k) {
    const int y = y0 - 2 + k;
    ov[k] = Dv[k] = 0.f;
    if (in_x && y >= 0 && y < H) {
      const int i = y * W + px;
      ov[k] = __ldg(im.opac + i);
      Dv[k] = __ldg(im.depth + i);
    }
  }
  // kAhead: the other inputs too, N_r of rows y0 - 1 .. y0 + R and the colours
  // and observed depths of the strip's own
  F3 nr_in[kAhead ? R + 2 : 1], rgb_in[kAhead ? R : 1], obs_in[kAhead ? R : 1];
  float od_in[kAhead ? R : 1];
  auto rgb_at = [](const float* p, int i) {
    return f3(__ldg(p + 3 * i), __ldg(p + 3 * i + 1), __ldg(p + 3 * i + 2));
  };
  if (kAhead) {
#pragma unroll
    for (int k = 0; k < R + 2; ++k) {
      const int y = y0 - 1 + k;
      nr_in[k] = f3(0.f, 0.f, 0.f);
      if (in_x && y >= 0 && y < H) nr_in[k] = rgb_at(im.normal, y * W + px);
    }
#pragma unroll
    for (int k = 0; k < R; ++k) {
      const int i = (y0 + k) * W + px;
      if (out_x && y0 + k < H) {
        rgb_in[k] = rgb_at(im.rgb, i);
        obs_in[k] = rgb_at(im.obs_rgb, i);
        od_in[k] = __ldg(im.obs_depth + i);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < kR; ++k) dv[k] = Dv[k] / fmaxf(ov[k], 1e-6f);
  // row q = e - 1: its normal term, dL_n / dN_r and dL_n / dX from its left
  // and right stencils; and the vertical part of row q - 1
  bool ok_q = false, ok_u = false;
  float ln_q = 0.f;
  F3 gn_q = f3(0.f, 0.f, 0.f), hx_q = gn_q, gy_q = gn_q, gy_u = gn_q;
  float acc = 0.f;
#pragma unroll
  for (int k = 1; k < kR - 1; ++k) {
    const int e = y0 - 2 + k;
    const float du = dv[k - 1], dc = dv[k], dd = dv[k + 1];   // rows e - 1, e, e + 1
    const float ou = ov[k - 1], oc = ov[k], od = ov[k + 1];
    // the normal term at (px, e): false if invalid (border pixel, own or a
    // 4-neighbour's opacity <= 0.5, degenerate cross product)
    const float dl = __shfl_up_sync(0xffffffffu, dc, 1), dr = __shfl_down_sync(0xffffffffu, dc, 1);
    const float ol = __shfl_up_sync(0xffffffffu, oc, 1), orr = __shfl_down_sync(0xffffffffu, oc, 1);
    bool ok = false;
    float Ln = 0.f;
    F3 gNr = f3(0.f, 0.f, 0.f), ggx = gNr, ggy = gNr;
    if (lane >= 1 && lane <= 30 && px >= 1 && e >= 1 && px <= W - 2 && e <= H - 2 && oc > 0.5f &&
        ol > 0.5f && orr > 0.5f && ou > 0.5f && od > 0.5f) {
      const int i = e * W + px;
      const float ryu = ((e - 1) + 0.5f - cam.cy) * ify, ryc = (e + 0.5f - cam.cy) * ify,
                  ryd = ((e + 1) + 0.5f - cam.cy) * ify;
      // half the differences of the neighbours' back-projected points
      const F3 gx = 0.5f * f3(fmaf(dr, rxr, -__fmul_rn(dl, rxl)), fmaf(dr, ryc, -__fmul_rn(dl, ryc)),
                              dr - dl);
      const F3 gy = 0.5f * f3(fmaf(dd, rxc, -__fmul_rn(du, rxc)), fmaf(dd, ryd, -__fmul_rn(du, ryu)),
                              dd - du);
      const F3 n = cross_rn(gx, gy);
      const float n2 = dot3(n, n);
      if (n2 > 0.f) {
        ok = true;
        const float inn = rsqrtf(n2);  // 1 / |n|
        const F3 ND = inn * n;
        const F3 Nr = kAhead ? nr_in[kAhead ? k - 1 : 0] : rgb_at(im.normal, i);
        const float dp = dot3(ND, Nr);
        Ln = 1.f - dp;
        gNr = (-1.f) * ND;
        // dLn/dn = -(Nr - ND (ND . Nr)) / |n|
        const F3 gn = (-inn) * f3(fmaf(-dp, ND.x, Nr.x), fmaf(-dp, ND.y, Nr.y), fmaf(-dp, ND.z, Nr.z));
        // dL_n / dX(p + ex) = 0.5 ggx, of X(p - ex) the negative; ggy alike
        ggx = cross_rn(gy, gn);
        ggy = cross_rn(gn, gx);
      }
    }
    // dL_n / dX(px, e) from the stencils of the left (uses X(p + ex)) and
    // right (X(p - ex)) neighbours
    const bool okl = __shfl_up_sync(0xffffffffu, (int)ok, 1) != 0;
    const bool okr = __shfl_down_sync(0xffffffffu, (int)ok, 1) != 0;
    const F3 gl = f3(__shfl_up_sync(0xffffffffu, ggx.x, 1), __shfl_up_sync(0xffffffffu, ggx.y, 1),
                     __shfl_up_sync(0xffffffffu, ggx.z, 1));
    const F3 gr = f3(__shfl_down_sync(0xffffffffu, ggx.x, 1),
                     __shfl_down_sync(0xffffffffu, ggx.y, 1),
                     __shfl_down_sync(0xffffffffu, ggx.z, 1));
    F3 hx = f3(0.f, 0.f, 0.f);
    if (okl) hx = fma_rn(0.5f, gl, hx);
    if (okr) hx = fma_rn(-0.5f, gr, hx);
    const int q = e - 1;
    if (k >= 3 && q < H && out_x) {
      const int i = q * W + px;
      const float O = ou, Dh = du;
      const float Oc = fmaxf(O, 1e-6f);
      const float D = Dv[k - 1];
      const int own = kAhead ? k - 3 : 0;   // the strip's row
      const F3 cr = kAhead ? rgb_in[own] : rgb_at(im.rgb, i);
      const F3 co = kAhead ? obs_in[own] : rgb_at(im.obs_rgb, i);
      const float d0 = cr.x - co.x, d1 = cr.y - co.y, d2 = cr.z - co.z;
      const float ddp = Dh - (kAhead ? od_in[own] : __ldg(im.obs_depth + i));
      acc += fmaf(w_l1, fabsf(d0) + fabsf(d1) + fabsf(d2), __fmul_rn(w_d, fabsf(ddp)));
      const float sl = w_l1 * inv;
      im.g_rgb[3 * i] = sgnf(d0) * sl;
      im.g_rgb[3 * i + 1] = sgnf(d1) * sl;
      im.g_rgb[3 * i + 2] = sgnf(d2) * sl;
      float gDh = __fmul_rn(w_d * sgnf(ddp), inv);
      // own normal term
      if (ok_q) acc = fmaf(w_n, ln_q, acc);
      const float sn = w_n * inv;
      im.g_normal[3 * i] = sn * gn_q.x;
      im.g_normal[3 * i + 1] = sn * gn_q.y;
      im.g_normal[3 * i + 2] = sn * gn_q.z;
      // and the stencils above (uses X(p + ey)) and below (X(p - ey))
      F3 gX = hx_q;
      if (ok_u) gX = fma_rn(0.5f, gy_u, gX);
      if (ok) gX = fma_rn(-0.5f, ggy, gX);
      const F3 rq = f3(rxc, (q + 0.5f - cam.cy) * ify, 1.f);
      gDh = fmaf(sn, dot3(gX, rq), gDh);
      im.g_depth[i] = gDh / Oc;
      im.g_opac[i] = O > 1e-6f ? -gDh * D / (O * O) : 0.f;
    }
    ok_u = ok_q;
    gy_u = gy_q;
    ok_q = ok;
    ln_q = Ln;
    gn_q = gNr;
    hx_q = hx;
    gy_q = ggy;
  }
  return acc;
}

template <int R>
__global__ void __launch_bounds__(kLossThreads, loss_blocks_per_sm(R, kLossThreads)) mapping_loss_kernel(
    MapLossImages im, gs2d_camera cam, float w_l1, float w_d, float w_n,
    float* __restrict__ part) {
  __shared__ float s[kLossWarps];
  const int strips_x = strips_along(cam.width, kStripW);
  const int n = strips_x * strips_along(cam.height, R);
  const float inv = 1.f / (float)(cam.width * cam.height);
  const float ifx = 1.f / cam.fx, ify = 1.f / cam.fy;
  float acc = 0.f;
  for (int k = blockIdx.x * kLossWarps + (threadIdx.x >> 5); k < n; k += gridDim.x * kLossWarps)
    acc += mapping_loss_strip<R>((k % strips_x) * kStripW, (k / strips_x) * R, im, cam, ifx,
                              ify, inv, w_l1, w_d, w_n);
  const float t = block_sum256(acc, s);
  if (threadIdx.x == 0) part[blockIdx.x] = t * inv;
}

// The mapping loss of many views in one launch: work items are the views'
// strips in view order; each strip's loss terms are summed over its warp
// into part[item], and mapping_loss_batch_sum_kernel adds each view's items
// in order.
struct LossViewDev {
  gs2d_camera cam;
  MapLossImages im;
  int strips_x, item0, n_items;
};
struct LossTable {
  int n_views, n_items;
  LossViewDev v[GS2D_MAX_VIEWS];
};

template <int R>
__global__ void __launch_bounds__(batch_threads(R), loss_blocks_per_sm(R, batch_threads(R)))
    mapping_loss_batch_kernel(const LossTable tab, float w_d, float w_n, float* __restrict__ part) {
  constexpr int kWarps = batch_threads(R) / 32;
  for (int item = blockIdx.x * kWarps + (threadIdx.x >> 5); item < tab.n_items;
       item += gridDim.x * kWarps) {
    int v = 0;
    while (v + 1 < tab.n_views && item >= tab.v[v + 1].item0) ++v;
    const LossViewDev& V = tab.v[v];
    const int k = item - V.item0;
    const float inv = 1.f / (float)(V.cam.width * V.cam.height);
    float acc = mapping_loss_strip<R>((k % V.strips_x) * kStripW, (k / V.strips_x) * R, V.im,
                                   V.cam, 1.f / V.cam.fx, 1.f / V.cam.fy, inv, 1.f, w_d, w_n);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0) part[item] = acc;
  }
}

// loss_out[v] = inv_v x the sum of view v's strip partials: thread t adds
// entries t, t + 256, ... in order, then a fixed tree over the threads.
__global__ void __launch_bounds__(256) mapping_loss_batch_sum_kernel(const LossTable tab,
                                                                     const float* __restrict__ part,
                                                                     float* __restrict__ loss_out) {
  __shared__ float s[256];
  const LossViewDev& V = tab.v[blockIdx.x];
  const float* p = part + V.item0;
  const int n = V.n_items;
  float a = 0.f;
#pragma unroll 8
  for (int e = threadIdx.x; e < n; e += 256) a += p[e];
  s[threadIdx.x] = a;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h) s[threadIdx.x] += s[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) loss_out[blockIdx.x] = s[0] / (float)(V.cam.width * V.cam.height);
}

size_t loss_ws_bytes(const gs2d_camera* cam) {
  (void)cam;
  return align_up(kLossBlocks * sizeof(float), 256);
}

int tracking_loss_launch(const float* rgb, const float* depth, const float* normal,
                         const float* opacity, const float* obs_rgb, const float* obs_depth,
                         const gs2d_camera* cam, const gs2d_track_params* prm, float* g_rgb,
                         float* g_depth, float* g_opacity, float* loss_out, void* workspace,
                         size_t ws_bytes, size_t* ws_needed, const int32_t* gate, cudaStream_t st) {
  if (!rgb || !depth || !normal || !opacity || !obs_rgb || !obs_depth || !cam || !prm || !g_rgb ||
      !g_depth || !g_opacity || !loss_out)
    return GS2D_ERR_INVALID_ARG;
  if (cam->width <= 0 || cam->height <= 0) return GS2D_ERR_INVALID_ARG;
  const size_t need = loss_ws_bytes(cam);
  if (ws_needed) *ws_needed = need;
  if (!workspace || ws_bytes < need) return GS2D_ERR_WORKSPACE;
  float* part = static_cast<float*>(workspace);
  tracking_loss_kernel<<<kLossBlocks, kLossThreads, 0, st>>>(rgb, depth, normal, opacity, obs_rgb,
                                                             obs_depth, *cam, *prm, g_rgb, g_depth,
                                                             g_opacity, part, gate);
  GS2D_LAUNCH_CHECK();
  sum_parts_kernel<<<1, 256, 0, st>>>(part, kLossBlocks, loss_out, gate);
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

}  // namespace gs2d

using namespace gs2d;

extern "C" {

int gs2d_tracking_loss(const float* rgb, const float* depth, const float* normal,
                       const float* opacity, const float* obs_rgb, const float* obs_depth,
                       const gs2d_camera* cam, const gs2d_track_params* prm, float* g_rgb,
                       float* g_depth, float* g_opacity, float* loss_out, void* workspace,
                       size_t ws_bytes, size_t* ws_needed, gs2d_stream stream) {
  return tracking_loss_launch(rgb, depth, normal, opacity, obs_rgb, obs_depth, cam, prm, g_rgb,
                              g_depth, g_opacity, loss_out, workspace, ws_bytes, ws_needed, nullptr,
                              (cudaStream_t)stream);
}

int gs2d_mapping_loss(const float* rgb, const float* depth, const float* normal,
                      const float* opacity, const float* obs_rgb, const float* obs_depth,
                      const gs2d_camera* cam, float w_d, float w_n, float* g_rgb, float* g_depth,
                      float* g_normal, float* g_opacity, float* loss_out, void* workspace,
                      size_t ws_bytes, size_t* ws_needed, gs2d_stream stream) {
  return gs2d_mapping_loss_ssim(rgb, depth, normal, opacity, obs_rgb, obs_depth, cam, 0.f, w_d,
                                w_n, g_rgb, g_depth, g_normal, g_opacity, loss_out, workspace,
                                ws_bytes, ws_needed, stream);
}

size_t gs2d_mapping_loss_batch_workspace(const gs2d_loss_view* views, int n_views) {
  if (!views || n_views <= 0 || n_views > GS2D_MAX_VIEWS) return 0;
  size_t items = 0;
  for (int v = 0; v < n_views; ++v) {
    const gs2d_camera& c = views[v].cam;
    if (c.width <= 0 || c.height <= 0) return 0;
    // eight partials per 32 x 8 pixels: room for the smaller strips (28 x 2) of
    // any size, ceil(w / 28) <= 2 ceil(w / 32) and ceil(h / 2) <= 4 ceil(h / 8)
    items += (size_t)strips_along(c.width, 32) * strips_along(c.height, 8) * 8;
  }
  return align_up(items * sizeof(float), 256);
}

int gs2d_mapping_loss_batch(const gs2d_loss_view* views, int n_views, float w_d, float w_n,
                            float* loss_out, void* workspace, size_t ws_bytes, size_t* ws_needed,
                            gs2d_stream stream) {
  if (!views || n_views <= 0 || n_views > GS2D_MAX_VIEWS || !loss_out) return GS2D_ERR_INVALID_ARG;
  LossTable tab;
  tab.n_views = n_views;
  long long items = 0, px = 0;
  for (int v = 0; v < n_views; ++v) px += (long long)views[v].cam.width * views[v].cam.height;
  const int rows = strip_rows(px);
  for (int v = 0; v < n_views; ++v) {
    const gs2d_loss_view& x = views[v];
    if (!x.rgb || !x.depth || !x.normal || !x.opacity || !x.obs_rgb || !x.obs_depth || !x.g_rgb ||
        !x.g_depth || !x.g_normal || !x.g_opacity)
      return GS2D_ERR_INVALID_ARG;
    if (x.cam.width <= 0 || x.cam.height <= 0) return GS2D_ERR_INVALID_ARG;
    LossViewDev& d = tab.v[v];
    d.cam = x.cam;
    d.im = MapLossImages{x.rgb,     x.depth, x.normal,  x.opacity,  x.obs_rgb,
                         x.obs_depth, x.g_rgb, x.g_depth, x.g_normal, x.g_opacity};
    d.strips_x = strips_along(x.cam.width, kStripW);
    d.item0 = (int)items;
    const long long mine = (long long)d.strips_x * strips_along(x.cam.height, rows);
    d.n_items = (int)mine;
    items += mine;
    // an int counts strips, past the last one by at most a grid's stride
    if (items > 0x7FFFFFFF - (1 << 20)) return GS2D_ERR_INVALID_ARG;
  }
  tab.n_items = (int)items;
  const size_t need = gs2d_mapping_loss_batch_workspace(views, n_views);
  if (ws_needed) *ws_needed = need;
  if (!workspace || ws_bytes < need) return GS2D_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  float* part = static_cast<float*>(workspace);
  // a resident grid, or every strip's block (the partials are per item, so
  // the result does not depend on it)
  static int slots[64] = {};
  int dev = 0;
  GS2D_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return GS2D_ERR_CUDA;
  if (!slots[dev]) {
    int sms = 0;
    GS2D_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    slots[dev] = loss_blocks_per_sm(kStripRows, kLossThreads) * max(1, sms);
  }
  if (rows == kStripRows) {
    const int blocks = min(slots[dev], strips_along(tab.n_items, kLossWarps));
    mapping_loss_batch_kernel<kStripRows><<<blocks, kLossThreads, 0, st>>>(tab, w_d, w_n, part);
  } else {
    constexpr int kThreads = batch_threads(kStripRowsSmall);
    mapping_loss_batch_kernel<kStripRowsSmall>
        <<<strips_along(tab.n_items, kThreads / 32), kThreads, 0, st>>>(tab, w_d, w_n, part);
  }
  GS2D_LAUNCH_CHECK();
  mapping_loss_batch_sum_kernel<<<n_views, 256, 0, st>>>(tab, part, loss_out);
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

size_t gs2d_mapping_loss_ssim_workspace(const gs2d_camera* cam) {
  if (!cam || cam->width <= 0 || cam->height <= 0) return 0;
  return loss_ws_bytes(cam) + ssim_ws_bytes(cam->height, cam->width);
}

int gs2d_mapping_loss_ssim(const float* rgb, const float* depth, const float* normal,
                           const float* opacity, const float* obs_rgb, const float* obs_depth,
                           const gs2d_camera* cam, float w_ssim, float w_d, float w_n,
                           float* g_rgb, float* g_depth, float* g_normal, float* g_opacity,
                           float* loss_out, void* workspace, size_t ws_bytes, size_t* ws_needed,
                           gs2d_stream stream) {
  if (!rgb || !depth || !normal || !opacity || !obs_rgb || !obs_depth || !cam || !g_rgb ||
      !g_depth || !g_normal || !g_opacity || !loss_out)
    return GS2D_ERR_INVALID_ARG;
  if (cam->width <= 0 || cam->height <= 0 || !(w_ssim >= 0.f && w_ssim <= 1.f))
    return GS2D_ERR_INVALID_ARG;
  const size_t base = loss_ws_bytes(cam);
  const size_t need = w_ssim > 0.f ? base + ssim_ws_bytes(cam->height, cam->width) : base;
  if (ws_needed) *ws_needed = need;
  if (!workspace || ws_bytes < need) return GS2D_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  float* part = static_cast<float*>(workspace);
  const int rows = strip_rows((long long)cam->width * cam->height);
  const int strips = strips_along(cam->width, kStripW) * strips_along(cam->height, rows);
  const int blocks = min(kLossBlocks, strips_along(strips, kLossWarps));
  const MapLossImages im{rgb,     depth, normal,  opacity,  obs_rgb,
                         obs_depth, g_rgb, g_depth, g_normal, g_opacity};
  if (rows == kStripRows)
    mapping_loss_kernel<kStripRows><<<blocks, kLossThreads, 0, st>>>(im, *cam, 1.f - w_ssim, w_d,
                                                                     w_n, part);
  else
    mapping_loss_kernel<kStripRowsSmall><<<blocks, kLossThreads, 0, st>>>(im, *cam, 1.f - w_ssim,
                                                                          w_d, w_n, part);
  GS2D_LAUNCH_CHECK();
  sum_parts_kernel<<<1, 256, 0, st>>>(part, blocks, loss_out, nullptr);
  GS2D_LAUNCH_CHECK();
  if (w_ssim > 0.f)
    return ssim_launch(rgb, obs_rgb, cam->height, cam->width, w_ssim, g_rgb, loss_out,
                       static_cast<char*>(workspace) + base, ws_bytes - base, nullptr, st);
  return GS2D_OK;
}

}  // extern "C"
