// gs2d_render_fwd / gs2d_render_bwd: tile-based front-to-back compositing of
// 2D Gaussian surfels (Eq. alpha_blending) and its reverse mode to the surfel
// parameters and to the camera pose (Sec. III-B, Eq. derivatives), plus the
// fused tracking kernel (forward, tracking loss and pose backward per tile).
//
// Forward: one 256-thread block per image tile, one pixel per thread, each
// warp an 8 x 4 pixel block.  The tile's depth-ordered surfel list is staged
// through shared memory in batches of 256 records, the record's linear
// intersection map re-based on the tile's first pixel (c0t); a warp skips a
// surfel whose footprint misses its block, and every thread evaluates
// u = p0/p2, v = p1/p2, z = det/p2 with p = c0t + lx c1 + ly c2,
// G = exp(-(u^2+v^2)/2), a = min(alpha G, alpha_max), skips a < alpha_min or
// u^2+v^2 > cutoff or z <= near, blends colour, depth z, normal t_nc and
// opacity, and stops before the transmittance would fall below t_min.  The
// block leaves the list once every pixel has stopped.
//
// Backward: each pixel replays its list back to front from the stored
// (T_final, n_last): T_i = T_{i+1} / (1 - a_i), and with the running suffix
// S = sum_{j>i} w_j (c_j . gC + z_j gD + t_nc,j . gN) the blending gradient is
//   dL/da_i = T_i (c_i . gC + z_i gD + t_nc,i . gN) - (S - gO T_final) / (1 - a_i).
// Through the intersection, with q = gu d_u + gv d_v (dual tangents) and
// beta = (q . r + gz) / (n . r) (r the pixel ray, n = m_u x m_v), the
// gradient of one (pixel, surfel) pair w.r.t. the camera-space splat is
// rank one:
//   dL/dmu_c = Gv,  dL/d(s_u t_uc) = u Gv,  dL/d(s_v t_vc) = v Gv,  Gv = beta n - q,
// (moving the plane along n shifts the hit point along the ray; moving it
// in-plane shifts (u, v) through the dual basis).  The left pose perturbation
// moves every splat by (rho, theta x .), so the pair's pose gradient is
// (Gv, X x Gv) with X = z r the hit point, plus t_nc x dL/dt_nc from the
// normal image -- the Jacobians [I, -mu_c^x] and [0, -R_c,:,i^x] of Sec. III-B
// contracted with these rank-one gradients.
//
// Full mode: one warp replays one region of a tile (bwd_warp.cuh) and writes a
// 64-byte partial per (tile, region, surfel) at the pair's emission index.  A
// second kernel adds each surfel's partials in emission order
// (deterministic), chains to world space, scales and the quaternion, and
// forms the pose term.
// Tracking mode: pixels accumulate the 6-vector pose gradient directly; one
// partial per tile, reduced in a fixed order.
#include <type_traits>

#include "bwd_warp.cuh"
#include "gs2d_common.cuh"
#include "gs2d_internal.h"
#include "loss_pixel.cuh"
#include "quad.cuh"
#include "tile_loops.cuh"
#include "tile_sort.cuh"
#include "track_update.cuh"

namespace gs2d {

// Blocks per SM of the tile kernels with P pixels per thread.
template <int P>
constexpr int tile_blocks_per_sm() {
  return P == 1 ? 4 : (P == 2 ? 3 : 2);
}

template <bool kCount, int P>
__global__ void __launch_bounds__(kTileThreads, tile_blocks_per_sm<P>()) render_fwd_kernel(
    const float4* __restrict__ proj, const uint32_t* __restrict__ vals,
    const int32_t* __restrict__ ranges, gs2d_camera cam, gs2d_config cfg, int tiles_x,
    float* __restrict__ out_rgb, float* __restrict__ out_depth, float* __restrict__ out_normal,
    float* __restrict__ out_opac, float* __restrict__ out_T, uint32_t* __restrict__ out_nlast,
    unsigned long long* __restrict__ counts, const int32_t* __restrict__ gate) {
  __shared__ float4 s_rec[kTileThreads][kFwdVec4];
  __shared__ HitLists hl;
  if (gate && *gate) return;
  const int tile = blockIdx.x;
  const TilePix<P> tp = tile_pixel<P>(tile, tiles_x, cfg.tile_w, cfg.tile_h);
  bool inside[P];
#pragma unroll
  for (int k = 0; k < P; ++k) inside[k] = tp.px < cam.width && tp.py + 4 * k < cam.height;
  const int tile_x0 = (tile % tiles_x) * cfg.tile_w, tile_y0 = (tile / tiles_x) * cfg.tile_h;
  const float xt = (float)tile_x0 + 0.5f - cam.cx;
  const float yt = (float)tile_y0 + 0.5f - cam.cy;
  uint32_t cnt[5] = {0u, 0u, 0u, 0u, 0u};
  FwdState st[P];
  fwd_tile<kFwdVec4, kCount, P>(proj, vals + ranges[2 * tile], ranges[2 * tile], ranges[2 * tile + 1], xt, yt,
                                    tile_x0, tile_y0, tp, inside, cam, cfg, s_rec, hl, cnt, st);
  if (kCount) {
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      unsigned long long v = cnt[k];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
      if ((threadIdx.x & 31) == 0) atomicAdd(counts + k, v);
    }
    return;
  }
#pragma unroll
  for (int k = 0; k < P; ++k) {
    if (!inside[k]) continue;
    const size_t p = (size_t)(tp.py + 4 * k) * cam.width + tp.px;
    out_rgb[3 * p] = st[k].C.x;
    out_rgb[3 * p + 1] = st[k].C.y;
    out_rgb[3 * p + 2] = st[k].C.z;
    out_depth[p] = st[k].D;
    out_normal[3 * p] = st[k].N.x;
    out_normal[3 * p + 1] = st[k].N.y;
    out_normal[3 * p + 2] = st[k].N.z;
    out_opac[p] = 1.f - st[k].T;
    out_T[p] = st[k].T;
    out_nlast[p] = st[k].last;
  }
}

// The forward pass on 8 x 8 quadrants (quad.cuh), four blocks per tile: the
// tile's sorted list in batches of 256 positions, the entries that touch the
// quadrant staged in order.
__global__ void __launch_bounds__(kTileThreads, 4) render_fwd_quad_kernel(
    const float4* __restrict__ proj, const uint32_t* __restrict__ vals,
    const int32_t* __restrict__ ranges, gs2d_camera cam, gs2d_config cfg, int tiles_x,
    float* __restrict__ out_rgb, float* __restrict__ out_depth, float* __restrict__ out_normal,
    float* __restrict__ out_opac, float* __restrict__ out_T, uint32_t* __restrict__ out_nlast,
    const int32_t* __restrict__ gate) {
  __shared__ QuadStage<kFwdVec4> s;
  __shared__ uint8_t s_pos[kQuadBatch];       // list position within the batch of a staged entry
  __shared__ int s_cnt[2][kTileThreads / 32];
  if (gate && *gate) return;
  const int tile = blockIdx.x / kQuads, q = blockIdx.x % kQuads;
  const int tile_x0 = (tile % tiles_x) * cfg.tile_w, tile_y0 = (tile / tiles_x) * cfg.tile_h;
  const QuadPix tp = quad_pixel(q, tile_x0, tile_y0, cfg.tile_w, quad_flat(cfg));
  const bool inside = tp.px < cam.width && tp.py < cam.height;
  const float xt = (float)tile_x0 + 0.5f - cam.cx;
  const float yt = (float)tile_y0 + 0.5f - cam.cy;
  const int start = ranges[2 * tile], end = ranges[2 * tile + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  QuadFwd st = quad_fwd_init(inside);
  // the next batch's ids are in flight while this one is blended
  int idx = start + (int)threadIdx.x;
  uint32_t id = idx < end ? vals[idx] : 0u;
  for (int b = start, turn = 0; b < end; b += kQuadBatch, turn ^= 1) {
    uint32_t m = 0u;
    if (idx < end) {
      const float4 r7 = proj[(size_t)id * (kProjFloats / 4) + 7];
      m = quad_mask(r7.z, r7.w, tp);
    }
    const uint32_t bal = __ballot_sync(0xffffffffu, m != 0u);
    if (lane == 0) s_cnt[turn][warp] = __popc(bal);
    // also: the previous batch is no longer read
    if (__syncthreads_count(!st.done) == 0) break;
    int at = __popc(bal & ((1u << lane) - 1u)), n = 0;
#pragma unroll
    for (int w = 0; w < kTileThreads / 32; ++w) {
      const int c = s_cnt[turn][w];
      if (w < warp) at += c;
      n += c;
    }
    if (m) {
      stage_record_to<kFwdVec4>(proj, id, xt, yt, s.rec[at]);
      s.mask[at] = (uint8_t)m;
      s_pos[at] = (uint8_t)threadIdx.x;
    }
    idx += kQuadBatch;
    id = idx < end ? vals[idx] : 0u;
    __syncthreads();
    const int nh = quad_hits(s, n);
    quad_blend(s, nh, tp, cam, cfg, st,
               [&](int j) { return (uint32_t)(b - start + s_pos[j] + 1); });
  }
  if (!inside) return;
  const size_t p = (size_t)tp.py * cam.width + tp.px;
  switch (lane & 3) {   // each lane its components of the pixel
    case 0:
      out_rgb[3 * p] = st.a0;
      out_rgb[3 * p + 1] = st.a1;
      out_opac[p] = 1.f - st.T;
      break;
    case 1:
      out_rgb[3 * p + 2] = st.a0;
      out_depth[p] = st.a1;
      out_T[p] = st.T;
      break;
    case 2:
      out_normal[3 * p] = st.a0;
      out_normal[3 * p + 1] = st.a1;
      out_nlast[p] = st.last;
      break;
    default:
      out_normal[3 * p + 2] = st.a0;
      break;
  }
}

// Upstream gradients and compositing state of the thread's P pixels.
template <int P>
__device__ __forceinline__ void load_pix_grads(const TilePix<P>& tp, const bool (&inside)[P],
                                               const gs2d_camera& cam, const float* T_final,
                                               const uint32_t* n_last, const float* g_rgb,
                                               const float* g_depth, const float* g_normal,
                                               const float* g_opac, PixGrad (&pg)[P]) {
#pragma unroll
  for (int k = 0; k < P; ++k) {
    pg[k].Tf = 1.f;
    pg[k].nl = 0;
    pg[k].gC = f3(0.f, 0.f, 0.f);
    pg[k].gN = f3(0.f, 0.f, 0.f);
    pg[k].gD = 0.f;
    pg[k].gO = 0.f;
    if (!inside[k]) continue;
    const size_t p = (size_t)(tp.py + 4 * k) * cam.width + tp.px;
    pg[k].Tf = T_final[p];
    pg[k].nl = n_last[p];
    pg[k].gC = f3(g_rgb[3 * p], g_rgb[3 * p + 1], g_rgb[3 * p + 2]);
    pg[k].gD = g_depth[p];
    if (g_normal) pg[k].gN = f3(g_normal[3 * p], g_normal[3 * p + 1], g_normal[3 * p + 2]);
    if (g_opac) pg[k].gO = g_opac[p];
  }
}

// Pose-only backward (the full backward is render_bwd_warp_kernel): the
// tile's pose 6-vector partial.
template <int P>
__global__ void __launch_bounds__(kTileThreads, P == 1 ? 4 : (P == 2 ? 3 : 2)) render_bwd_kernel(
    const float4* __restrict__ proj, const uint32_t* __restrict__ vals,
    const int32_t* __restrict__ ranges, gs2d_camera cam, gs2d_config cfg, int tiles_x,
    const float* __restrict__ T_final, const uint32_t* __restrict__ n_last,
    const float* __restrict__ g_rgb, const float* __restrict__ g_depth,
    const float* __restrict__ g_normal, const float* __restrict__ g_opac,
    float* __restrict__ pose_part, const int32_t* __restrict__ gate) {
  __shared__ BwdSmem sm;
  __shared__ HitLists hl;
  __shared__ float s_pose[kTileThreads / 32][6];
  if (gate && *gate) return;
  const int tile = blockIdx.x;
  const TilePix<P> tp = tile_pixel<P>(tile, tiles_x, cfg.tile_w, cfg.tile_h);
  bool inside[P];
#pragma unroll
  for (int k = 0; k < P; ++k) inside[k] = tp.px < cam.width && tp.py + 4 * k < cam.height;
  const int tile_x0 = (tile % tiles_x) * cfg.tile_w, tile_y0 = (tile / tiles_x) * cfg.tile_h;
  const float xt = (float)tile_x0 + 0.5f - cam.cx;
  const float yt = (float)tile_y0 + 0.5f - cam.cy;
  const float rx = (tp.px + 0.5f - cam.cx) / cam.fx, ry = (tp.py + 0.5f - cam.cy) / cam.fy;
  PixGrad pg[P];
  load_pix_grads<P>(tp, inside, cam, T_final, n_last, g_rgb, g_depth, g_normal, g_opac, pg);
  float pr[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if (g_normal)
    bwd_tile_pose<true, P>(proj, vals + ranges[2 * tile], ranges[2 * tile], ranges[2 * tile + 1], xt, yt, tile_x0,
                           tile_y0, tp, inside, rx, ry, cam, cfg, pg, sm, hl, pr);
  else
    bwd_tile_pose<false, P>(proj, vals + ranges[2 * tile], ranges[2 * tile], ranges[2 * tile + 1], xt, yt, tile_x0,
                            tile_y0, tp, inside, rx, ry, cam, cfg, pg, sm, hl, pr);
  block_sum6(pr, s_pose, pose_part + (size_t)tile * 6);
}

// Full backward: one warp per (tile, region) work item, kBwdWarps warps per
// block and no block barrier (bwd_warp.cuh).
template <int R>
__global__ void __launch_bounds__(kBwdWarps * 32, kBwdWarpBlocks) render_bwd_warp_kernel(
    const float4* __restrict__ proj, const uint32_t* __restrict__ vals,
    const uint32_t* __restrict__ emit, const int32_t* __restrict__ ranges, gs2d_camera cam,
    gs2d_config cfg, int tiles_x, int Q, int n_units, const float* __restrict__ T_final,
    const uint32_t* __restrict__ n_last, const float* __restrict__ g_rgb,
    const float* __restrict__ g_depth, const float* __restrict__ g_normal,
    const float* __restrict__ g_opac, float* __restrict__ partials,
    const int32_t* __restrict__ gate) {
  __shared__ WarpBwdSmem<R> sm[kBwdWarps];
  if (gate && *gate) return;
  const int warp = threadIdx.x >> 5;
  const int unit = blockIdx.x * kBwdWarps + warp;
  if (unit >= n_units) return;
  const int tile = unit / Q, region = unit - tile * Q;
  bwd_region<R>(proj, vals, emit, ranges[2 * tile], ranges[2 * tile + 1],
                         (tile % tiles_x) * cfg.tile_w, (tile / tiles_x) * cfg.tile_h, region, Q,
                         cam, cfg, T_final, n_last, g_rgb, g_depth, g_normal, g_opac, partials,
                         sm[warp]);
}

// Shared memory of a fused tracking block that runs a whole tile.
struct TrackSmem {
  BwdSmem b;
  HitLists hl;
  float pose[kTileThreads / 32][6];
  float loss[kTileThreads / 32];
  uint32_t ids[kSegSmem];
};

// The ids of n sorted keys, clamped below n_ids.
__device__ __forceinline__ void key_ids(const unsigned long long* keys, int n, uint32_t* ids,
                                        int n_ids) {
  for (int i = threadIdx.x; i < n; i += kTileThreads)
    ids[i] = min((uint32_t)(keys[i] & 0xFFFFFFFFull), (uint32_t)(n_ids - 1));
  __syncthreads();
}

// The same for n <= kRankKeys unsorted, distinct keys: a key's place is its
// rank, counted by its own thread -- one pass and one barrier, where the runs
// and merges of the sort have four to six at these lengths.  The keys are
// visible to the block and 16-byte aligned.  40 iterations of whole tiles at
// 640x480, 26,400 surfels: 1895 -> 1770 us with the launch rule below; lists
// cut off at 64, 128 or 256 keys measure alike.
constexpr int kRankKeys = 256;
__device__ __forceinline__ void rank_ids(const unsigned long long* keys, int n, uint32_t* ids,
                                         int n_ids) {
  static_assert(kRankKeys <= kTileThreads, "a key per thread");
  if ((int)threadIdx.x < n) {
    const unsigned long long k = keys[threadIdx.x];
    int rank = 0, j = 0;
    for (; j + 1 < n; j += 2) {
      const ulonglong2 kk = *reinterpret_cast<const ulonglong2*>(keys + j);
      rank += (int)(kk.x < k) + (int)(kk.y < k);
    }
    if (j < n) rank += (int)(keys[j] < k);
    ids[rank] = min((uint32_t)(k & 0xFFFFFFFFull), (uint32_t)(n_ids - 1));
  }
  __syncthreads();
}

// Fused tracking iteration on one tile: the depth sort of the tile's
// segment, forward compositing, the tracking loss and its image gradient per
// pixel (in registers), and the pose-only backward replay -- the images never
// leave the chip.  Writes the tile's loss partial (already divided by
// |Omega|) and pose 6-vector partial.  A segment of at most kSegSmem keys is
// sorted in shared memory and its ids stay there; a longer one is sorted in
// chunks merged in global memory and its ids written to vals, which this
// block then reads back (coherent loads: vals is written in this launch).
// The block's per-warp sums end up in s.pose and s.loss (not yet visible to
// the other warps).
template <int P>
__device__ __forceinline__ void track_tile(
    int tile, const float4* __restrict__ proj, uint32_t* vals, const int32_t* __restrict__ ranges,
    const gs2d_camera& cam, const gs2d_config& cfg, int tiles_x,
    const float* __restrict__ obs_rgb, const float* __restrict__ obs_depth,
    const gs2d_track_params& prm, const TrackStep& ts, TrackSmem& s) {
  BwdSmem& sm = s.b;
  HitLists& hl = s.hl;
  uint32_t* s_ids = s.ids;
  const TilePix<P> tp = tile_pixel<P>(tile, tiles_x, cfg.tile_w, cfg.tile_h);
  bool inside[P];
#pragma unroll
  for (int k = 0; k < P; ++k) inside[k] = tp.px < cam.width && tp.py + 4 * k < cam.height;
  const int tile_x0 = (tile % tiles_x) * cfg.tile_w, tile_y0 = (tile / tiles_x) * cfg.tile_h;
  const float xt = (float)tile_x0 + 0.5f - cam.cx;
  const float yt = (float)tile_y0 + 0.5f - cam.cy;
  const float rx = (tp.px + 0.5f - cam.cx) / cam.fx, ry = (tp.py + 0.5f - cam.cy) / cam.fy;
  const int start = ranges[2 * tile], end = ranges[2 * tile + 1];
  // the segment's depth order, keys (depth bits << 32 | id) sorted in the
  // record staging area before any record is staged
  const uint32_t* ids;
  {
    const int len = end - start;
    unsigned long long* keys = reinterpret_cast<unsigned long long*>(&sm.rec[0][0]);
    static_assert(sizeof(sm.rec) >= kSegSmem * sizeof(unsigned long long), "sort area");
    constexpr int kTwice = (int)(sizeof(sm.rec) / (2 * sizeof(unsigned long long)));
    if (len <= kSegSmem) {
      for (int i = threadIdx.x; i < len; i += kTileThreads) keys[i] = ts.seg_keys[start + i];
      __syncthreads();
      if (len <= kRankKeys) {
        rank_ids(keys, len, s_ids, ts.n);
      } else {
        if (len <= kTwice)   // room for two copies
          keys = merge_sort(keys, keys + kTwice, len);
        else
          bitonic_sort(keys, len);
        key_ids(keys, len, s_ids, ts.n);
      }
      ids = s_ids;
    } else {
      sort_long_segment<kSegSmem>(tile, proj, ts.n, tiles_x, ranges, ts.seg_keys, ts.seg_tmp,
                                  nullptr, vals, nullptr, nullptr, (long long)end, keys);
      __syncthreads();
      ids = vals + start;
    }
  }
  FwdState st[P];
  fwd_tile<kBwdVec4, false, P>(proj, ids, start, end, xt, yt, tile_x0, tile_y0, tp, inside,
                                   cam, cfg, sm.rec, hl, nullptr, st);
  float pr[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  const float inv = 1.f / (float)(cam.width * cam.height);
  PixGrad pg[P];
  float loss = 0.f;
#pragma unroll
  for (int k = 0; k < P; ++k) {
    PixLoss L;
    L.loss = 0.f;
    L.g_rgb[0] = L.g_rgb[1] = L.g_rgb[2] = 0.f;
    L.g_depth = L.g_opac = 0.f;
    if (inside[k]) {
      const size_t p = (size_t)(tp.py + 4 * k) * cam.width + tp.px;
      L = tracking_pixel_loss(st[k].C, st[k].D, st[k].N, 1.f - st[k].T,
                              f3(obs_rgb[3 * p], obs_rgb[3 * p + 1], obs_rgb[3 * p + 2]),
                              obs_depth[p], rx, ry + (4.f * k) / cam.fy, inv, prm);
    }
    loss += L.loss * inv;
    pg[k].Tf = st[k].T;
    pg[k].nl = st[k].last;
    pg[k].gC = f3(L.g_rgb[0], L.g_rgb[1], L.g_rgb[2]);
    pg[k].gN = f3(0.f, 0.f, 0.f);
    pg[k].gD = L.g_depth;
    pg[k].gO = L.g_opac;
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, off);
  if ((threadIdx.x & 31) == 0) s.loss[threadIdx.x >> 5] = loss;
  // a list of at most one batch is still staged with its hit lists
  bwd_tile_pose<false, P>(proj, ids, start, end, xt, yt, tile_x0, tile_y0, tp, inside, rx, ry,
                              cam, cfg, pg, sm, hl, pr, end - start <= kTileThreads);
  warp_sum6(pr, s.pose);
}

// The last block of a fused tracking launch to finish reduces the tiles'
// partials and updates the pose.
__device__ __forceinline__ void track_finish(const float* pose_part, const float* loss_part,
                                             int n_tiles, const TrackStep& ts,
                                             const gs2d_track_params& prm, int32_t* status,
                                             bool* s_last, float (*s_red)[256]) {
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) *s_last = atomicAdd(ts.counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!*s_last) return;
  __threadfence();
  reduce_and_step(pose_part, loss_part, n_tiles, ts.pose, ts.adam, prm, ts.loss_hist,
                  ts.pose_hist, ts.grad_hist, ts.iter, status, s_red);
  if (threadIdx.x == 0) *ts.counter = 0u;
  // the next iteration's binning starts from zeroed counters (its kernels
  // run after this one; this iteration's binning finished before it)
  if (ts.sort_zero)
    for (size_t i = threadIdx.x; i < ts.sort_zero_words; i += blockDim.x) ts.sort_zero[i] = 0u;
}

// The tile's partial from its warps' sums, added in warp order.
__device__ __forceinline__ void write_tile_partial(const TrackSmem& s, int tile, float* pose_part,
                                                   float* loss_part) {
  __syncthreads();
  if (threadIdx.x < 7) {
    float v = 0.f;
    for (int w = 0; w < kTileThreads / 32; ++w)
      v += threadIdx.x < 6 ? s.pose[w][threadIdx.x] : s.loss[w];
    if (threadIdx.x < 6)
      pose_part[(size_t)tile * 6 + threadIdx.x] = v;
    else
      loss_part[tile] = v;
  }
}

// Whether the launch's status lets the block run; records the history of an
// iteration skipped after convergence.
__device__ __forceinline__ bool track_runs(const TrackStep& ts, const int32_t* status) {
  const int32_t g = *status;
  if (g == kConverged && blockIdx.x == 0 && threadIdx.x == 0)
    record_converged(ts.pose, ts.loss_hist, ts.pose_hist, ts.grad_hist, ts.iter);
  return g == 0;
}

template <int P>
__global__ void __launch_bounds__(kTileThreads, tile_blocks_per_sm<P>()) track_tile_kernel(
    const float4* __restrict__ proj, uint32_t* vals,
    const int32_t* __restrict__ ranges, gs2d_camera cam, gs2d_config cfg, int tiles_x,
    const float* __restrict__ obs_rgb, const float* __restrict__ obs_depth, gs2d_track_params prm,
    float* __restrict__ loss_part, float* __restrict__ pose_part, TrackStep ts,
    int32_t* __restrict__ status) {
  __shared__ TrackSmem s;
  __shared__ bool s_last;
  if (!track_runs(ts, status)) return;
  // longest lists first: the blocks of the heaviest tiles start in the first
  // wave instead of trailing the grid (partials stay indexed by tile)
  const int tile = ts.order ? ts.order[blockIdx.x] : (int)blockIdx.x;
  track_tile<P>(tile, proj, vals, ranges, cam, cfg, tiles_x, obs_rgb, obs_depth, prm, ts, s);
  write_tile_partial(s, tile, pose_part, loss_part);
  // 7 x 256 floats fit
  track_finish(pose_part, loss_part, gridDim.x, ts, prm, status, &s_last,
               reinterpret_cast<float(*)[256]>(&s.b.rec[0][0]));
}

// The fused iteration with one pixel per thread, tile by tile or on 8 x 8
// quadrants (quad.cuh): a quadrant's block takes the keys of its tile's
// segment whose footprint touches the quadrant, sorts them, blends, evaluates
// the loss and replays.  The first `split` tiles of the launch order have four
// blocks each (three of them leave at once when their tile runs whole), the
// others one; SplitRule says where the line lies.  Segments of more than
// kQuadKeys keys run whole, and maps of few surfels do not come here at all.
// A quadrant writes one partial per 8 x 4 pixel block and the last of the
// tile's four blocks adds the eight up in the whole-tile form's order, so the
// results do not depend on the choice.
constexpr int kQuadKeys = 3072;
struct QuadTrackSmem {
  union {
    QuadStage<kBwdVec4> st;
    unsigned long long keys[kQuadKeys];
  };
  uint32_t ids[kQuadKeys];
  float out[7][64];     // per pixel: the pose 6-vector and the loss
  int cnt;
};
constexpr int kTileParts = kTileThreads / 32;   // 8 x 4 blocks (partials) per tile

// Which tiles run on quadrants.  Four blocks finish a tile in a third of the
// time one takes, with about twice the instructions in all, so they pay where
// a tile would outlast the rest of the launch: where its list is longer than
// per_slot x K, the mean share of the K entries per resident block slot times
// a constant, and than min_len (below it the fixed cost of a block, ~15 us,
// is most of a tile's time).  Measured over 10 iterations, whole tiles alone
// -> this rule (three poses each, us):
//   160x120 (80 tiles), 200k surfels   2088-2649 -> 734-1219
//   320x240 (300 tiles), 200k surfels  1086-1742 -> 938-1075
//   480x360 (690 tiles), 200k surfels   973-1464 -> 964-1015
//   640x480 (1200 tiles), 200k surfels 1087-1366 -> 1099-1254
//   320x240 (300 tiles), 50k surfels    423-620  -> 417-523
// Up to two tiles per SM every tile may split and the other three blocks of
// each follow the tiles (their early exits then cost nothing where no tile
// splits); in larger grids only the half of the SM count longest tiles may,
// and their blocks lead the launch, so that they overlap the whole of it.
//
// Maps of few surfels for the grid have no lists worth splitting, and
// track_quad_kernel then costs more than track_tile_kernel<1>: its blocks that
// only leave, and more code to fetch.  Up to the line, 8,000 surfels and 30 more
// a tile, whole tiles were no slower at any grid; 40 iterations, us, whole
// tiles -> quadrants (median of three maps) at 0.6 / 1 / 1.5 / 2.2 times its
// surfels:
//   160x120   1234 -> 1249  1315 -> 1328  1413 -> 1412  1707 -> 1586
//   320x240   1328 -> 1400  1455 -> 1487  1592 -> 1644  1853 -> 1789
//   480x360   1498 -> 1538  1740 -> 1805  1985 -> 2033  2298 -> 2246
//   640x480   1770 -> 1847  2159 -> 2277  2470 -> 2574  2961 -> 3074
struct SplitRule {
  int split;         // tiles (in launch order) that may run on quadrants
  int extras_first;  // their four blocks each lead the grid
  int min_len;
  float per_slot;
};

__global__ void __launch_bounds__(kTileThreads, 4) track_quad_kernel(
    const float4* __restrict__ proj, uint32_t* vals,
    const int32_t* __restrict__ ranges, const int32_t* __restrict__ n_isect, gs2d_camera cam,
    gs2d_config cfg, int tiles_x, int n_tiles,
    const float* __restrict__ obs_rgb, const float* __restrict__ obs_depth, gs2d_track_params prm,
    float* __restrict__ loss_part, float* __restrict__ pose_part, SplitRule rule, TrackStep ts,
    int32_t* __restrict__ status) {
  __shared__ union Smem {
    QuadTrackSmem q;
    TrackSmem t;
    float red[7][256];
    __device__ Smem() {}
  } sh;
  __shared__ bool s_last;
  if (!track_runs(ts, status)) return;
  const int b0 = (int)blockIdx.x;
  int rank, quad;
  if (rule.extras_first) {
    const int rest = b0 - kQuads * rule.split;
    rank = rest < 0 ? b0 / kQuads : rule.split + rest;
    quad = rest < 0 ? b0 % kQuads : 0;
  } else {
    const int extra = b0 - n_tiles;
    rank = extra < 0 ? b0 : extra / (kQuads - 1);
    quad = extra < 0 ? 0 : 1 + extra % (kQuads - 1);
  }
  const int tile = ts.order[rank];
  const int start = ranges[2 * tile], end = ranges[2 * tile + 1], len = end - start;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool on_quads = rank < rule.split && len > rule.min_len && len <= kQuadKeys &&
                        (float)len > rule.per_slot * (float)*n_isect;
  if (!on_quads) {
    if (quad == 0) {
      track_tile<1>(tile, proj, vals, ranges, cam, cfg, tiles_x, obs_rgb, obs_depth, prm, ts, sh.t);
      write_tile_partial(sh.t, tile, pose_part, loss_part);
    }
  } else {
    QuadTrackSmem& s = sh.q;
    const int tile_x0 = (tile % tiles_x) * cfg.tile_w, tile_y0 = (tile / tiles_x) * cfg.tile_h;
    const QuadPix tp = quad_pixel(quad, tile_x0, tile_y0, cfg.tile_w, quad_flat(cfg));
    const bool inside = tp.px < cam.width && tp.py < cam.height;
    const float xt = (float)tile_x0 + 0.5f - cam.cx;
    const float yt = (float)tile_y0 + 0.5f - cam.cy;
    const float rx = (tp.px + 0.5f - cam.cx) / cam.fx, ry = (tp.py + 0.5f - cam.cy) / cam.fy;
    // the quadrant's keys, in any order
    if (threadIdx.x == 0) s.cnt = 0;
    __syncthreads();
    for (int i0 = 0; i0 < len; i0 += kTileThreads) {
      const int i = i0 + (int)threadIdx.x;
      unsigned long long key = 0ull;
      bool hit = false;
      if (i < len) {
        key = ts.seg_keys[start + i];
        const uint32_t id = min((uint32_t)(key & 0xFFFFFFFFull), (uint32_t)(ts.n - 1));
        const float4 r7 = proj[(size_t)id * (kProjFloats / 4) + 7];
        hit = quad_mask(r7.z, r7.w, tp) != 0u;
      }
      const uint32_t b = __ballot_sync(0xffffffffu, hit);
      int o = 0;
      if (lane == 0 && b) o = atomicAdd(&s.cnt, __popc(b));
      o = __shfl_sync(0xffffffffu, o, 0);
      if (hit) s.keys[o + __popc(b & ((1u << lane) - 1u))] = key;
    }
    __syncthreads();
    const int n = s.cnt;
    if (n <= kRankKeys) {
      rank_ids(s.keys, n, s.ids, ts.n);
    } else {
      unsigned long long* sorted = s.keys;
      if (n <= kQuadKeys / 2)   // room for two copies
        sorted = merge_sort(s.keys, s.keys + kQuadKeys / 2, n);
      else
        bitonic_sort(s.keys, n);
      key_ids(sorted, n, s.ids, ts.n);
    }
    auto stage = [&](int b, int cnt) {   // entries b .. b + cnt - 1; returns the warp's hits
      if ((int)threadIdx.x < cnt) {
        stage_record_to<kBwdVec4>(proj, s.ids[b + threadIdx.x], xt, yt, s.st.rec[threadIdx.x]);
        const float4 r6 = s.st.rec[threadIdx.x][6];
        s.st.mask[threadIdx.x] = (uint8_t)quad_mask(r6.z, r6.w, tp);
      }
      __syncthreads();
      return quad_hits(s.st, cnt);
    };
    QuadFwd st = quad_fwd_init(inside);
    int nh = 0, staged = 0;   // the batch in shared memory
    for (int b = 0; b < n; b += kQuadBatch) {
      if (__syncthreads_count(!st.done) == 0) break;
      nh = stage(b, min(kQuadBatch, n - b));
      staged = b;
      quad_blend(s.st, nh, tp, cam, cfg, st, [&](int j) { return (uint32_t)(b + j + 1); });
    }
    const QuadOut o = quad_gather(st);
    const float inv = 1.f / (float)(cam.width * cam.height);
    PixLoss L;
    L.loss = 0.f;
    L.g_rgb[0] = L.g_rgb[1] = L.g_rgb[2] = 0.f;
    L.g_depth = L.g_opac = 0.f;
    if (inside) {
      const size_t p = (size_t)tp.py * cam.width + tp.px;
      L = tracking_pixel_loss(o.C, o.D, o.N, 1.f - st.T,
                              f3(obs_rgb[3 * p], obs_rgb[3 * p + 1], obs_rgb[3 * p + 2]),
                              obs_depth[p], rx, ry, inv, prm);
    }
    PixGrad pg;
    pg.Tf = st.T;
    pg.nl = st.last;
    pg.gC = f3(L.g_rgb[0], L.g_rgb[1], L.g_rgb[2]);
    pg.gN = f3(0.f, 0.f, 0.f);
    pg.gD = L.g_depth;
    pg.gO = L.g_opac;
    QuadBwd bw;
    bw.T = st.T;
    bw.acc = 0.f;
    bw.sG = bw.szG = f3(0.f, 0.f, 0.f);
    for (int b = staged; b >= 0 && n > 0; b -= kQuadBatch) {
      if (b != staged) {
        __syncthreads();
        nh = stage(b, kQuadBatch);
      }
      quad_replay(s.st, nh, b, tp, cam, cfg, pg, rx, ry, cam.fx * cam.fy, bw);
    }
    const F3 th = cross3(f3(rx, ry, 1.f), bw.szG);
    if ((lane & 3) == 0) {
      s.out[0][tp.slot] = bw.sG.x;
      s.out[1][tp.slot] = bw.sG.y;
      s.out[2][tp.slot] = bw.sG.z;
      s.out[3][tp.slot] = th.x;
      s.out[4][tp.slot] = th.y;
      s.out[5][tp.slot] = th.z;
      s.out[6][tp.slot] = L.loss * inv;
    }
    __syncthreads();
    // the quadrant's two 8 x 4 blocks, each summed over its lanes as a warp
    // of the plain form sums them
    for (int v = warp; v < 14; v += kTileThreads / 32) {
      const int c = v >> 1, half = v & 1;
      float x = s.out[c][32 * half + lane];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
      const size_t part =
          (size_t)rank * kTileParts + quad_block(quad, half, cfg.tile_w, tp.flat);
      if (lane == 0) ts.quad_part[part * 7 + c] = x;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s.cnt = (int)atomicAdd(ts.quad_done + rank, 1u);
    __syncthreads();
    if (s.cnt == kQuads - 1) {
      __threadfence();
      if (threadIdx.x < 7) {
        float v = 0.f;
        for (int w = 0; w < kTileParts; ++w)
          v += __ldcg(ts.quad_part + ((size_t)rank * kTileParts + w) * 7 + threadIdx.x);
        if (threadIdx.x < 6)
          pose_part[(size_t)tile * 6 + threadIdx.x] = v;
        else
          loss_part[tile] = v;
      }
      if (threadIdx.x == 0) ts.quad_done[rank] = 0u;   // for the next iteration
    }
  }
  track_finish(pose_part, loss_part, n_tiles, ts, prm, status, &s_last, sh.red);
}

// Per-surfel reduction of the (tile, region, surfel) partials in emission
// order (Q region slots per tile) and the chain rule to world-space
// parameters, for one or several views of the same m records (record i is
// surfel active[i], or i); the views' gradients are summed in registers and
// written (or added) once.  Pose term per view and block.
//
// The sums are latency-bound gathers: a surfel's partials are contiguous, but
// a thread per surfel touches 32 places in a warp's load and leaves the lanes
// of surfels that the view does not see idle (half of them or more).  So a
// warp lists its surfels that have tiles and gives four lanes to each, a
// 16-byte quarter of every partial to a lane, eight surfels at a time; the
// sums then return to the surfel's own thread through shared memory for the
// chain rule.  1M surfels x 8 views of 1200 x 680: 684 -> 311 us (all
// views in one launch); 32 views of subsets, each in a launch of its own that
// mostly moves the scattered outputs and parameters, 1389 -> 1370 us.
// SPW: surfels per warp (grad_surfels_per_warp).
constexpr int kGradThreads = 256, kGradWarps = kGradThreads / 32;
template <int SPW>
__global__ void __launch_bounds__(kGradThreads, 3) surfel_grad_kernel(
    const GradTable t, const float* __restrict__ mu, const float* __restrict__ quat,
    const float* __restrict__ scale, int m, const int32_t* __restrict__ active, int n_all, int mode,
    int Q, float* __restrict__ d_mu, float* __restrict__ d_quat, float* __restrict__ d_scale,
    float* __restrict__ d_opac, float* __restrict__ d_rgb) {
  __shared__ float s_S[kGradWarps][32][kRedVals + 1];
  __shared__ unsigned char s_list[kGradWarps][32];
  __shared__ float s_in[GS2D_MAX_VIEWS][12];
  __shared__ float s_pose[GS2D_MAX_VIEWS][kGradWarps][6];
  __shared__ bool s_dead[GS2D_MAX_VIEWS];
  if (mode == kGradWrite && t.v[0].gate && *t.v[0].gate) return;
  for (int e = threadIdx.x; e < t.n * 12; e += kGradThreads) s_in[e / 12][e % 12] = t.v[e / 12].pose[e % 12];
  for (int v = threadIdx.x; v < t.n; v += kGradThreads) s_dead[v] = t.v[v].gate && *t.v[v].gate;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = ((int)blockIdx.x * kGradWarps + warp) * SPW + lane;
  const bool in = lane < SPW && i < m;
  const int sid = !in ? 0 : (active ? min(max(active[i], 0), n_all - 1) : i);
  float4 q4 = make_float4(1.f, 0.f, 0.f, 0.f);
  F3 mw = f3(0.f, 0.f, 0.f);
  float su = 0.f, sv = 0.f;
  if (in) {
    q4 = reinterpret_cast<const float4*>(quat)[sid];
    mw = f3(mu[3 * sid], mu[3 * sid + 1], mu[3 * sid + 2]);
    su = scale[2 * sid];
    sv = scale[2 * sid + 1];
  }
  // a view's counts and offsets are read one view ahead, whatever its gate says
  auto first_at = [&](int v, int& k, uint32_t& off) {
    const bool on = v < t.n && in;
    k = on ? t.v[v].tiles[i] * Q : 0;
    off = on ? t.v[v].surfel_off[i] : 0u;
  };
  int k_next;
  uint32_t off_next;
  first_at(0, k_next, off_next);
  __syncthreads();
  const float qn2 = fmaf(q4.x, q4.x, fmaf(q4.y, q4.y, fmaf(q4.z, q4.z, q4.w * q4.w)));
  const float qinv = rsqrtf(qn2);
  const float w = q4.x * qinv, x = q4.y * qinv, y = q4.z * qinv, z = q4.w * qinv;
  float a_scale[2] = {0.f, 0.f}, a_opac = 0.f, a_rgb[3] = {0.f, 0.f, 0.f};
  float a_mu[3] = {0.f, 0.f, 0.f}, a_quat[4] = {0.f, 0.f, 0.f, 0.f};
  bool any = mode != kGradAdd;
  for (int v = 0; v < t.n; ++v) {
    const GradView& V = t.v[v];
    const int k = s_dead[v] ? 0 : k_next;
    const uint32_t off = off_next;
    first_at(v + 1, k_next, off_next);
    const float* R = s_in[v];
    const F3 mu_c = mat_mul(R, mw) + f3(R[9], R[10], R[11]);
    // no sums and every factor of the chain finite: nothing to add (a factor
    // that is not finite makes the gradients NaN, as the products would)
    const float mag = fabsf(mu_c.x) + fabsf(mu_c.y) + fabsf(mu_c.z) + fabsf(su) + fabsf(sv) + qinv + qn2;
    const bool work = in && !s_dead[v] && (k > 0 || !(mag < __int_as_float(0x7f800000)));
    const unsigned has = __ballot_sync(0xffffffffu, k > 0);
    const float4* rec = reinterpret_cast<const float4*>(V.proj) + (size_t)i * (kProjFloats / 4);
    if (k > 0) {
      asm volatile("prefetch.global.L1 [%0];" ::"l"(rec + 2));
      asm volatile("prefetch.global.L1 [%0];" ::"l"(rec + 4));
      asm volatile("prefetch.global.L1 [%0];" ::"l"(rec + 6));
      s_list[warp][__popc(has & ((1u << lane) - 1u))] = (unsigned char)lane;
    }
    __syncwarp();
    const int n_has = __popc(has);
    for (int j0 = 0; j0 < n_has; j0 += 8) {
      const int j = j0 + (lane >> 2);
      const int src = s_list[warp][min(j, n_has - 1)];
      int kk = __shfl_sync(0xffffffffu, k, src);
      const uint32_t oo = __shfl_sync(0xffffffffu, off, src);
      if (j >= n_has) kk = 0;
      const float4* p = reinterpret_cast<const float4*>(V.partials) + (size_t)oo * Q * 4 + (lane & 3);
      float4 S = make_float4(0.f, 0.f, 0.f, 0.f);
      int kk_max = kk;
#pragma unroll
      for (int o = 16; o > 2; o >>= 1) kk_max = max(kk_max, __shfl_xor_sync(0xffffffffu, kk_max, o));
      for (int e = 0; e < kk_max; e += 8, p += 32) {
        float4 t[8];
#pragma unroll
        for (int c = 0; c < 4; ++c) t[c] = e + c < kk ? p[4 * c] : make_float4(0.f, 0.f, 0.f, 0.f);
        if (e + 4 < kk_max)
#pragma unroll
          for (int c = 4; c < 8; ++c) t[c] = e + c < kk ? p[4 * c] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int c = 0; c < 4; ++c) S.x += t[c].x, S.y += t[c].y, S.z += t[c].z, S.w += t[c].w;
        if (e + 4 < kk_max)
#pragma unroll
          for (int c = 4; c < 8; ++c) S.x += t[c].x, S.y += t[c].y, S.z += t[c].z, S.w += t[c].w;
      }
      if (j < n_has) {
        float* o = &s_S[warp][src][4 * (lane & 3)];
        o[0] = S.x, o[1] = S.y, o[2] = S.z, o[3] = S.w;
      }
    }
    __syncwarp();
    float pr[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (work) {
      any = true;
      const F3 tu = f3(1.f - 2.f * (y * y + z * z), 2.f * (x * y + w * z), 2.f * (x * z - w * y));
      const F3 tv = f3(2.f * (x * y - w * z), 1.f - 2.f * (x * x + z * z), 2.f * (y * z + w * x));
      const F3 tn = f3(2.f * (x * z + w * y), 2.f * (y * z - w * x), 1.f - 2.f * (x * x + y * y));
      const F3 tuc = mat_mul(R, tu), tvc = mat_mul(R, tv), tnc = mat_mul(R, tn);
      // sum Gv, sum u Gv, sum v Gv from the moment sums and the record's
      // n, d_u, d_v and opacity (a surfel in no tile has all sums zero)
      F3 g_muc = f3(0.f, 0.f, 0.f), g_mu = g_muc, g_mv = g_muc, g_tnc = g_muc;
      if (k > 0) {
        const float* S = s_S[warp][lane];
        const float4 r2 = rec[2], r4 = rec[4], r5 = rec[5], r6 = rec[6];
        // record floats 17..25 (n, d_u, d_v) and 10 (opacity)
        const F3 nrm = f3(r4.y, r4.z, r4.w), du = f3(r5.x, r5.y, r5.z), dv = f3(r5.w, r6.x, r6.y);
        const float op = r2.z;
        g_muc = S[0] * nrm + op * (S[4] * du + S[5] * dv);
        g_mu = S[1] * nrm + op * (S[6] * du + S[7] * dv);
        g_mv = S[2] * nrm + op * (S[7] * du + S[8] * dv);
        g_tnc = f3(S[12], S[13], S[14]);
        a_opac += S[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) a_rgb[c] += S[9 + c];
      }
      const F3 g_tuc = su * g_mu, g_tvc = sv * g_mv;
      a_scale[0] += dot3(tuc, g_mu);
      a_scale[1] += dot3(tvc, g_mv);
      const F3 th = cross3(mu_c, g_muc) + cross3(tuc, g_tuc) + cross3(tvc, g_tvc) + cross3(tnc, g_tnc);
      pr[0] = g_muc.x; pr[1] = g_muc.y; pr[2] = g_muc.z;
      pr[3] = th.x; pr[4] = th.y; pr[5] = th.z;
      const F3 gmw = mat_tmul(R, g_muc);
      a_mu[0] += gmw.x, a_mu[1] += gmw.y, a_mu[2] += gmw.z;
      // world-space column gradients G[:,0..2] = R^T g_t{u,v,n}c
      const F3 G0 = mat_tmul(R, g_tuc), G1 = mat_tmul(R, g_tvc), G2 = mat_tmul(R, g_tnc);
      // d/dq of the rotation matrix of a unit quaternion, contracted with G
      // (G_rc = gradient of entry (r, c); column c of R is t_u, t_v, t_n)
      const float G00 = G0.x, G10 = G0.y, G20 = G0.z;
      const float G01 = G1.x, G11 = G1.y, G21 = G1.z;
      const float G02 = G2.x, G12 = G2.y, G22 = G2.z;
      const float gw = 2.f * (z * (G10 - G01) + y * (G02 - G20) + x * (G21 - G12));
      const float gx = 2.f * (y * (G10 + G01) + z * (G02 + G20) + w * (G21 - G12)) - 4.f * x * (G11 + G22);
      const float gy = 2.f * (x * (G10 + G01) + z * (G12 + G21) + w * (G02 - G20)) - 4.f * y * (G00 + G22);
      const float gz = 2.f * (x * (G02 + G20) + y * (G12 + G21) + w * (G10 - G01)) - 4.f * z * (G00 + G11);
      // unit quaternion -> raw quaternion: (I - q q^T) / |q|
      const float qd = w * gw + x * gx + y * gy + z * gz;
      a_quat[0] += (gw - w * qd) * qinv;
      a_quat[1] += (gx - x * qd) * qinv;
      a_quat[2] += (gy - y * qd) * qinv;
      a_quat[3] += (gz - z * qd) * qinv;
    }
    const bool warp_any = __any_sync(0xffffffffu, work);
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      float r = pr[c];
      if (warp_any)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
      if (lane == 0) s_pose[v][warp][c] = r;
    }
  }
  if (in && any) {
    // o(p, v): write, or add to what earlier launches left
    auto o = [&](float* p, float r) { *p = mode == kGradAdd ? *p + r : r; };
    o(d_scale + 2 * sid, a_scale[0]);
    o(d_scale + 2 * sid + 1, a_scale[1]);
    o(d_opac + sid, a_opac);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      o(d_rgb + 3 * sid + c, a_rgb[c]);
      o(d_mu + 3 * sid + c, a_mu[c]);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) o(d_quat + 4 * sid + c, a_quat[c]);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < t.n * 6; e += kGradThreads) {
    float r = 0.f;
    for (int ww = 0; ww < kGradWarps; ++ww) r += s_pose[e / 6][ww][e % 6];
    t.v[e / 6].pose_part[(size_t)blockIdx.x * 6 + e % 6] = r;
  }
}

// Fixed-order sum of per-block 6-vector partials, a view per block.
__global__ void __launch_bounds__(256) pose_reduce_kernel(const PoseReduceTable t) {
  __shared__ float s[6][256];
  const PoseReduceView& V = t.v[blockIdx.x];
  if (V.gate && *V.gate) return;
  const float* __restrict__ part = V.part;
  const int n_part = V.n_part;
  float acc[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
  for (int b = threadIdx.x; b < n_part; b += 256)
#pragma unroll
    for (int c = 0; c < 6; ++c) acc[c] += part[(size_t)b * 6 + c];
#pragma unroll
  for (int c = 0; c < 6; ++c) s[c][threadIdx.x] = acc[c];
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h)
#pragma unroll
      for (int c = 0; c < 6; ++c) s[c][threadIdx.x] += s[c][threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x < 6) V.out[threadIdx.x] = s[threadIdx.x][0];
}

struct BwdWs {
  float* partials;
  float* pose_part;
  size_t bytes;
};
BwdWs carve_bwd_ws(void* base, int n, size_t cap, int n_tiles, bool full, int Q) {
  Carver c(base);
  BwdWs w;
  w.partials = c.take<float>(full ? (cap > 0 ? cap : 1) * Q * kRedVals : 1);
  const int nb = max(n_tiles, grad_blocks_room(n));
  w.pose_part = c.take<float>((size_t)max(nb, 1) * 6);
  w.bytes = align_up(c.off, 256);
  return w;
}

int validate_tile_cfg(const gs2d_camera* cam, const gs2d_config* cfg) {
  if (!cam || !cfg) return GS2D_ERR_INVALID_ARG;
  // P pixels per thread; warps cover 8 x 4P pixel blocks of the tile
  if (!tile_cfg_ok(*cfg)) return GS2D_ERR_INVALID_ARG;
  if (cam->width <= 0 || cam->height <= 0) return GS2D_ERR_INVALID_ARG;
  const long long nt = (long long)gs2d_tiles_x(cam, cfg) * gs2d_tiles_y(cam, cfg);
  if (nt > 65535) return GS2D_ERR_INVALID_ARG;
  return GS2D_OK;
}

// gs2d_set_grouped_tiles: grids of at most this many tiles run on quadrants
// (quad.cuh); -1: the library's own rule.
static int g_grouped_max_tiles = -1;

static int sm_count() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 0;
  return sms;
}

// Whether the forward pass of a one-pixel grid of n_tiles tiles runs on
// quadrants: up to two tiles per SM.
static bool use_grouped(int px_per_thread, int n_tiles) {
  if (px_per_thread != 1) return false;
  return n_tiles <= (g_grouped_max_tiles < 0 ? 2 * sm_count() : g_grouped_max_tiles);
}

// Whether a tracking iteration over n surfels runs the kernel whose tiles may
// split (see SplitRule).
static bool track_splits(int n, int n_tiles) {
  if (g_grouped_max_tiles >= 0) return n_tiles <= g_grouped_max_tiles;
  return n > 8000 + 30 * n_tiles;
}

static SplitRule split_rule(int n_tiles) {
  if (g_grouped_max_tiles >= 0) return SplitRule{n_tiles, 0, 0, 0.f};
  const int sms = max(sm_count(), 1), slots = 4 * sms;
  if (n_tiles <= 2 * sms) return SplitRule{n_tiles, 0, 80, 1.25f / slots};
  return SplitRule{min(sms / 2, n_tiles), 1, 80, 1.75f / slots};
}

int render_fwd_launch(const float* proj, const gs2d_bins* bins, const gs2d_camera* cam,
                      const gs2d_config* cfg, float* rgb, float* depth, float* normal,
                      float* opacity, float* t_final, uint32_t* n_last, const int32_t* gate,
                      cudaStream_t st) {
  const int v = validate_tile_cfg(cam, cfg);
  if (v) return v;
  if (!proj || !bins || !bins->vals || !bins->tile_ranges || !rgb || !depth || !normal ||
      !opacity || !t_final || !n_last)
    return GS2D_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(proj) & 15) return GS2D_ERR_INVALID_ARG;
  const int tx = gs2d_tiles_x(cam, cfg), ty = gs2d_tiles_y(cam, cfg);
  if (use_grouped(cfg->px_per_thread, tx * ty))
    render_fwd_quad_kernel<<<tx * ty * kQuads, kTileThreads, 0, st>>>(
        reinterpret_cast<const float4*>(proj), bins->vals, bins->tile_ranges, *cam, *cfg, tx, rgb,
        depth, normal, opacity, t_final, n_last, gate);
  else
    GS2D_DISPATCH_P(cfg->px_per_thread, render_fwd_kernel<false, P><<<tx * ty, kTileThreads, 0, st>>>(
        reinterpret_cast<const float4*>(proj), bins->vals, bins->tile_ranges, *cam, *cfg, tx, rgb,
        depth, normal, opacity, t_final, n_last, nullptr, gate));
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

#define GS2D_TRACK_TILE(P)                                                                      \
  track_tile_kernel<P><<<tx * ty, kTileThreads, 0, st>>>(                                       \
      reinterpret_cast<const float4*>(proj), bins->vals, bins->tile_ranges, *cam, *cfg, tx,     \
      obs_rgb, obs_depth, *prm, loss_part, pose_part, ts, status)

int track_tile_launch(const float* proj, const gs2d_bins* bins, const gs2d_camera* cam,
                      const gs2d_config* cfg, const float* obs_rgb, const float* obs_depth,
                      const gs2d_track_params* prm, float* loss_part, float* pose_part,
                      const TrackStep& ts, int32_t* status, cudaStream_t st) {
  const int v = validate_tile_cfg(cam, cfg);
  if (v) return v;
  if (!proj || !bins || !bins->vals || !bins->tile_ranges || !obs_rgb || !obs_depth || !prm ||
      !loss_part || !pose_part || !ts.pose || !ts.adam || !ts.counter || !status)
    return GS2D_ERR_INVALID_ARG;
  const int tx = gs2d_tiles_x(cam, cfg), ty = gs2d_tiles_y(cam, cfg);
  if (cfg->px_per_thread == 1 && track_splits(ts.n, tx * ty)) {
    if (!bins->n_isect || !ts.order || !ts.quad_part || !ts.quad_done) return GS2D_ERR_INVALID_ARG;
    const SplitRule rule = split_rule(tx * ty);
    track_quad_kernel<<<tx * ty + (kQuads - 1) * rule.split, kTileThreads, 0, st>>>(
        reinterpret_cast<const float4*>(proj), bins->vals, bins->tile_ranges, bins->n_isect, *cam,
        *cfg, tx, tx * ty, obs_rgb, obs_depth, *prm, loss_part, pose_part, rule, ts, status);
  } else {
    switch (cfg->px_per_thread) {
      case 1: GS2D_TRACK_TILE(1); break;
      case 2: GS2D_TRACK_TILE(2); break;
      case 3: GS2D_TRACK_TILE(3); break;
      default: GS2D_TRACK_TILE(4); break;
    }
  }
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

int surfel_grad_launch(const gs2d_surfels* s, const int32_t* active, int m, int mode, int Q,
                       const GradTable& t, float* d_mu, float* d_quat, float* d_scale,
                       float* d_opac, float* d_rgb, cudaStream_t st) {
  if (m <= 0) return GS2D_OK;
  auto kern = grad_surfels_per_warp(m) == 8 ? surfel_grad_kernel<8> : surfel_grad_kernel<32>;
  kern<<<grad_blocks(m), kGradThreads, 0, st>>>(t, s->mu, s->quat, s->scale, m, active, s->n, mode, Q,
                                                d_mu, d_quat, d_scale, d_opac, d_rgb);
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

int pose_reduce_batch_launch(const PoseReduceTable& t, cudaStream_t st) {
  pose_reduce_kernel<<<t.n, 256, 0, st>>>(t);
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

// One view's pose reduction.
static int pose_reduce_one(const float* part, int n_part, float* out, const int32_t* gate,
                           cudaStream_t st) {
  PoseReduceTable t;
  t.n = 1;
  t.v[0] = PoseReduceView{part, n_part, out, gate};
  return pose_reduce_batch_launch(t, st);
}

size_t render_bwd_ws_bytes(int n, size_t cap, int n_tiles, bool full, int Q) {
  return carve_bwd_ws(nullptr, n, cap, n_tiles, full, Q).bytes;
}

int render_bwd_launch(const float* proj, const gs2d_bins* bins, const int32_t* tiles_per_surfel,
                      const gs2d_surfels* s, const float* pose, const gs2d_camera* cam,
                      const gs2d_config* cfg, const float* t_final, const uint32_t* n_last,
                      const float* d_rgb, const float* d_depth, const float* d_normal,
                      const float* d_opacity, float* d_mu, float* d_quat, float* d_scale,
                      float* d_opac, float* d_rgb_out, float* d_pose6, void* workspace,
                      size_t ws_bytes, size_t* ws_needed, const int32_t* gate, cudaStream_t st) {
  const int v = validate_tile_cfg(cam, cfg);
  if (v) return v;
  if (!proj || !bins || !bins->vals || !bins->tile_ranges || !t_final || !n_last || !d_rgb ||
      !d_depth || !s)
    return GS2D_ERR_INVALID_ARG;
  const bool any = d_mu || d_quat || d_scale || d_opac || d_rgb_out;
  const bool full = any;
  if (full && !(d_mu && d_quat && d_scale && d_opac && d_rgb_out)) return GS2D_ERR_INVALID_ARG;
  if (full && (!bins->isect_emit || !bins->surfel_off || !tiles_per_surfel || !s->mu ||
               !s->quat || !s->scale || !pose))
    return GS2D_ERR_INVALID_ARG;
  if (!full && !d_pose6) return GS2D_ERR_INVALID_ARG;
  const int tx = gs2d_tiles_x(cam, cfg), ty = gs2d_tiles_y(cam, cfg);
  const int n_tiles = tx * ty;
  // partials sized for the largest tile shape, so the size follows from
  // (n, capacity, n_tiles) alone
  const size_t need = render_bwd_ws_bytes(s->n, bins->capacity, n_tiles, full, kBwdMaxRegions);
  if (ws_needed) *ws_needed = need;
  if (!workspace || ws_bytes < need) return GS2D_ERR_WORKSPACE;
  const BwdWs w = carve_bwd_ws(workspace, s->n, bins->capacity, n_tiles, full, kBwdMaxRegions);
  const float4* p4 = reinterpret_cast<const float4*>(proj);
  if (full) {
    // regions as small as fill the GPU: see bwd_region_for
    const int R = bwd_region_for(*cfg, n_tiles);
    const int Q = bwd_regions(*cfg, R);
    const int units = n_tiles * Q;
    const int blocks = (units + kBwdWarps - 1) / kBwdWarps;
    auto launch = [&](auto r) {
      render_bwd_warp_kernel<decltype(r)::value><<<blocks, kBwdWarps * 32, 0, st>>>(
          p4, bins->vals, bins->isect_emit, bins->tile_ranges, *cam, *cfg, tx, Q, units, t_final,
          n_last, d_rgb, d_depth, d_normal, d_opacity, w.partials, gate);
    };
    if (R == 1)
      launch(std::integral_constant<int, 1>());
    else if (R == 2)
      launch(std::integral_constant<int, 2>());
    else if (R == 4)
      launch(std::integral_constant<int, 4>());
    else
      launch(std::integral_constant<int, kBwdRegion>());
    GS2D_LAUNCH_CHECK();
    if (s->n > 0) {
      GradTable t;
      t.n = 1;
      t.v[0] = GradView{pose, tiles_per_surfel, bins->surfel_off, proj, w.partials, w.pose_part, gate};
      const int gr = surfel_grad_launch(s, nullptr, s->n, kGradWrite, Q, t, d_mu, d_quat, d_scale,
                                        d_opac, d_rgb_out, st);
      if (gr) return gr;
      if (d_pose6) {
        const int pr = pose_reduce_one(w.pose_part, grad_blocks(s->n), d_pose6, gate, st);
        if (pr) return pr;
      }
    } else if (d_pose6) {
      GS2D_CUDA_TRY(cudaMemsetAsync(d_pose6, 0, 6 * sizeof(float), st));
    }
  } else {
    GS2D_DISPATCH_P(cfg->px_per_thread, render_bwd_kernel<P><<<n_tiles, kTileThreads, 0, st>>>(
        p4, bins->vals, bins->tile_ranges, *cam, *cfg, tx, t_final, n_last, d_rgb, d_depth,
        d_normal, d_opacity, w.pose_part, gate));
    GS2D_LAUNCH_CHECK();
    const int pr = pose_reduce_one(w.pose_part, n_tiles, d_pose6, gate, st);
    if (pr) return pr;
  }
  return GS2D_OK;
}

}  // namespace gs2d

using namespace gs2d;

extern "C" {

int gs2d_render_fwd(const float* proj, const gs2d_bins* bins, const gs2d_camera* cam,
                    const gs2d_config* cfg, float* rgb, float* depth, float* normal,
                    float* opacity, float* t_final, uint32_t* n_last, gs2d_stream stream) {
  if (!bins) return GS2D_ERR_INVALID_ARG;
  return render_fwd_launch(proj, bins, cam, cfg, rgb, depth, normal, opacity, t_final, n_last,
                           bins->status, (cudaStream_t)stream);
}

int gs2d_render_count(const float* proj, const gs2d_bins* bins, const gs2d_camera* cam,
                      const gs2d_config* cfg, unsigned long long* counts, gs2d_stream stream) {
  const int v = validate_tile_cfg(cam, cfg);
  if (v) return v;
  if (!proj || !bins || !bins->vals || !bins->tile_ranges || !counts) return GS2D_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  GS2D_CUDA_TRY(cudaMemsetAsync(counts, 0, 5 * sizeof(unsigned long long), st));
  const int tx = gs2d_tiles_x(cam, cfg), ty = gs2d_tiles_y(cam, cfg);
  GS2D_DISPATCH_P(cfg->px_per_thread, render_fwd_kernel<true, P><<<tx * ty, kTileThreads, 0, st>>>(
      reinterpret_cast<const float4*>(proj), bins->vals, bins->tile_ranges, *cam, *cfg, tx, nullptr,
      nullptr, nullptr, nullptr, nullptr, nullptr, counts, bins->status));
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

void gs2d_set_grouped_tiles(int max_tiles) { g_grouped_max_tiles = max_tiles < -1 ? -1 : max_tiles; }

size_t gs2d_render_bwd_workspace(int n, size_t capacity, int n_tiles) {
  return render_bwd_ws_bytes(n, capacity, n_tiles, true, kBwdMaxRegions);
}

int gs2d_render_bwd(const float* proj, const gs2d_bins* bins, const int32_t* tiles_per_surfel,
                    const gs2d_surfels* s, const float* pose, const gs2d_camera* cam,
                    const gs2d_config* cfg, const float* t_final, const uint32_t* n_last,
                    const float* d_rgb, const float* d_depth, const float* d_normal,
                    const float* d_opacity, float* d_mu, float* d_quat, float* d_scale,
                    float* d_opac, float* d_rgb_out, float* d_pose6, void* workspace,
                    size_t ws_bytes, size_t* ws_needed, gs2d_stream stream) {
  if (!bins) return GS2D_ERR_INVALID_ARG;
  return render_bwd_launch(proj, bins, tiles_per_surfel, s, pose, cam, cfg, t_final, n_last, d_rgb,
                           d_depth, d_normal, d_opacity, d_mu, d_quat, d_scale, d_opac, d_rgb_out,
                           d_pose6, workspace, ws_bytes, ws_needed, bins->status,
                           (cudaStream_t)stream);
}

}  // extern "C"
