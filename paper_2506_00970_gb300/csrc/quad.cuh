// Compositing of an 8 x 8 pixel quadrant by a 256-thread block: the form of
// the one-pixel tile loops (tile_loops.cuh) for tile grids too small to fill
// the GPU, where the serial walk of each pixel over its tile's list is the
// bound (160x120 has 80 tiles of 16x16; one thread per pixel leaves 1 warp
// per scheduler).
//
// A 256-pixel tile is cut into its four 8 x 8 quadrants, one block each (a tile
// of 64 x 4 pixels into four of 16 x 4).  The block keeps only the entries whose footprint touches its quadrant (about
// half of a small image's list), and each warp owns 4 x 2 pixels with four
// lanes per pixel (lane = 4 * pixel + e): the lanes evaluate four successive
// hits of their pixel at once, then all four replay the pixel's transmittance
// over them in list order -- every lane the same numbers -- while the sums are
// split over the lanes by component.  Evaluations, their order and every
// per-pixel sum are those of the plain loops, so images, losses and pose
// gradients are bit-identical to theirs.
//
// Against four evaluations in flight per thread over whole tiles (the form
// this replaces): four times the warps, half the evaluated pairs (a 4 x 2
// block of pixels misses more footprints than an 8 x 4 one) and half the
// entries to sort; the fused tracking kernel at 160x120, 200k surfels,
// 191 -> 81 us per iteration, the forward pass of the same view 62-101 ->
// 25-43 us.  Bound by the latency of the longest list's walk.
#pragma once

#include "tile_loops.cuh"

namespace gs2d {

constexpr int kQuads = 4;        // 8 x 8 quadrants of a 256-pixel tile
constexpr int kQuadBatch = 256;  // entries staged at a time

// Tiles 4 pixels high have quadrants of 16 x 4 pixels.
__device__ __forceinline__ bool quad_flat(const gs2d_config& cfg) { return cfg.tile_h < 8; }

// The block's quadrant and the lane's pixel: quadrant q at tile offset
// (8 (q % (tile_w / 8)), 8 (q / (tile_w / 8))), warp w the 4 x 2 pixels at
// (4 (w & 1), 2 (w >> 1)) of it; in a flat tile at (16 q, 0) and
// (4 (w & 3), 2 (w >> 2)).
struct QuadPix {
  int x0, y0;      // the quadrant's first pixel
  int px, py;      // the lane's pixel
  float lx, ly;    // its centre relative to the tile's first pixel centre
  int slot;        // its index in the quadrant, whose two 8 x 4 blocks follow each other
  bool flat;
};
__device__ __forceinline__ QuadPix quad_pixel(int q, int tile_x0, int tile_y0, int tile_w,
                                              bool flat) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, p = lane >> 2;
  const int per_row = tile_w >> 3;
  const int ox = flat ? q * 16 : (q % per_row) * 8, oy = flat ? 0 : (q / per_row) * 8;
  const int cx = (flat ? w & 3 : w & 1) * 4 + (p & 3), cy = (flat ? w >> 2 : w >> 1) * 2 + (p >> 2);
  QuadPix t;
  t.x0 = tile_x0 + ox;
  t.y0 = tile_y0 + oy;
  t.px = t.x0 + cx;
  t.py = t.y0 + cy;
  t.lx = (float)(ox + cx);
  t.ly = (float)(oy + cy);
  t.slot = flat ? 32 * (cx >> 3) + 8 * cy + (cx & 7) : 8 * cy + cx;
  t.flat = flat;
  return t;
}

// Which of the tile's 8 x 4 pixel blocks is block `half` of quadrant q.
__device__ __forceinline__ int quad_block(int q, int half, int tile_w, bool flat) {
  if (flat) return 2 * q + half;
  const int per_row = tile_w >> 3;
  return (2 * (q / per_row) + half) * per_row + q % per_row;
}

// Mask of the quadrant's eight warps whose 4 x 2 pixels a footprint (packed
// pixel ranges) touches; 0 when it misses the quadrant.
__device__ __forceinline__ uint32_t quad_mask(float bi, float bj, const QuadPix& tp) {
  const uint32_t I = __float_as_uint(bi), J = __float_as_uint(bj);
  const int i0 = max((int)(I & 0xFFFF) - tp.x0, 0);
  const int i1 = min((int)(I >> 16) - tp.x0, tp.flat ? 15 : 7);
  const int j0 = max((int)(J & 0xFFFF) - tp.y0, 0);
  const int j1 = min((int)(J >> 16) - tp.y0, tp.flat ? 3 : 7);
  if (i0 > i1 || j0 > j1) return 0u;
  if (tp.flat) {
    const uint32_t cols = (2u << (i1 >> 2)) - (1u << (i0 >> 2));
    return (j0 < 2 ? cols : 0u) | (j1 >= 2 ? cols << 4 : 0u);
  }
  const uint32_t cols = (i0 < 4 ? 1u : 0u) | (i1 >= 4 ? 2u : 0u);
  uint32_t m = 0u;
#pragma unroll
  for (int r = 0; r < 4; ++r)
    if (j1 >= 2 * r && j0 <= 2 * r + 1) m |= cols << (2 * r);
  return m;
}

// Staged entries of one batch.
template <int kStride>
struct QuadStage {
  float4 rec[kQuadBatch][kStride];
  uint8_t mask[kQuadBatch];
  uint8_t list[8][kQuadBatch];
};

// The warp's hits of a staged batch of n entries, in order.
template <int kStride>
__device__ __forceinline__ int quad_hits(QuadStage<kStride>& s, int n) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int nh = 0;
  for (int c = 0; c < n; c += 32) {
    const int j = c + lane;
    const bool hit = j < n && ((s.mask[j] >> warp) & 1u);
    const uint32_t b = __ballot_sync(0xffffffffu, hit);
    if (hit) s.list[warp][nh + __popc(b & ((1u << lane) - 1u))] = (uint8_t)j;
    nh += __popc(b);
  }
  __syncwarp();
  return nh;
}

// Forward state of the lane's pixel: T, last and done are the pixel's (the
// same in its four lanes), a0 and a1 the lane's two components of
//   e = 0: (C.x, C.y)   1: (C.z, D)   2: (N.x, N.y)   3: (N.z, -).
struct QuadFwd {
  float T, a0, a1;
  uint32_t last;
  bool done;
};
__device__ __forceinline__ QuadFwd quad_fwd_init(bool inside) {
  QuadFwd st;
  st.T = 1.f;
  st.a0 = st.a1 = 0.f;
  st.last = 0u;
  st.done = !inside;
  return st;
}

// Blends the warp's nh hits of a staged batch.  pos_of(j): one past the list
// position of staged entry j (what n_last counts).
template <int kStride, class Pos>
__device__ __forceinline__ void quad_blend(const QuadStage<kStride>& s, int nh, const QuadPix& tp,
                                           const gs2d_camera& cam, const gs2d_config& cfg,
                                           QuadFwd& st, Pos pos_of) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, e = lane & 3, base = lane & 28;
  // the lane's components in a staged record (floats 11..16: rgb, t_nc)
  const int wa = kRgb + (e == 0 ? 0 : e == 1 ? 2 : e == 2 ? 3 : 5), wb = e == 3 ? wa : wa + 1;
  for (int h0 = 0; h0 < nh; h0 += 4) {
    if (__all_sync(0xffffffffu, st.done)) break;
    const int j = s.list[warp][min(h0 + e, nh - 1)];
    Eval ev;
    const bool hit = eval_pair(s.rec[j][0], s.rec[j][1], s.rec[j][2], tp.lx, tp.ly, cam.near_z,
                               cfg.cutoff_r2, cfg.alpha_min, cfg.alpha_max, ev) &&
                     h0 + e < nh && !st.done;
    const uint32_t hits = __ballot_sync(0xffffffffu, hit);
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      if (!(hits & (0x11111111u << g))) continue;   // warp-uniform
      const float a = __shfl_sync(0xffffffffu, ev.a, base | g);
      const float z = __shfl_sync(0xffffffffu, ev.z, base | g);
      const int jg = __shfl_sync(0xffffffffu, j, g);   // the same entry for every pixel
      if (!((hits >> (base | g)) & 1u) || st.done) continue;
      const float Tn = st.T * (1.f - a);
      if (Tn < cfg.t_min) {
        st.done = true;
        continue;
      }
      const float* rec = reinterpret_cast<const float*>(s.rec[jg]);
      const float w = a * st.T;
      st.a0 = fmaf(w, rec[wa], st.a0);
      st.a1 = fmaf(w, e == 1 ? z : rec[wb], st.a1);
      st.T = Tn;
      st.last = pos_of(jg);
    }
    __syncwarp();
  }
}

// The pixel's eight outputs in all four lanes.
struct QuadOut {
  F3 C, N;
  float D;
};
__device__ __forceinline__ QuadOut quad_gather(const QuadFwd& st) {
  const int base = threadIdx.x & 28;
  QuadOut o;
  o.C.x = __shfl_sync(0xffffffffu, st.a0, base);
  o.C.y = __shfl_sync(0xffffffffu, st.a1, base);
  o.C.z = __shfl_sync(0xffffffffu, st.a0, base | 1);
  o.D = __shfl_sync(0xffffffffu, st.a1, base | 1);
  o.N.x = __shfl_sync(0xffffffffu, st.a0, base | 2);
  o.N.y = __shfl_sync(0xffffffffu, st.a1, base | 2);
  o.N.z = __shfl_sync(0xffffffffu, st.a0, base | 3);
  return o;
}

// Pose-only replay of the warp's nh hits of a staged batch, back to front
// (bwd_tile_pose without a normal gradient): b0 = the list position of the
// batch's first entry.  T, acc, sG and szG are the pixel's, the same in its
// four lanes.
struct QuadBwd {
  float T, acc;
  F3 sG, szG;
};
__device__ __forceinline__ void quad_replay(const QuadStage<kBwdVec4>& s, int nh, int b0,
                                            const QuadPix& tp, const gs2d_camera& cam,
                                            const gs2d_config& cfg, const PixGrad& pg, float rx,
                                            float ry, float fxfy, QuadBwd& st) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, e = lane & 3, base = lane & 28;
  const float gOT = pg.gO * pg.Tf;
  for (int h0 = nh - 1; h0 >= 0; h0 -= 4) {
    const int j = s.list[warp][max(h0 - e, 0)];
    const float4 r2 = s.rec[j][2];
    Eval ev;
    const bool hit = eval_pair(s.rec[j][0], s.rec[j][1], r2, tp.lx, tp.ly, cam.near_z,
                               cfg.cutoff_r2, cfg.alpha_min, cfg.alpha_max, ev) &&
                     h0 - e >= 0 && b0 + j < (int)pg.nl;
    const uint32_t hits = __ballot_sync(0xffffffffu, hit);
    if (!hits) continue;
    // the lane's own pair, as far as it needs no running state
    const float4 r3 = s.rec[j][3], r4 = s.rec[j][4], r5 = s.rec[j][5], r6 = s.rec[j][6];
    const float iom = rcp_ftz(1.f - ev.a);
    const float vj = fmaf(r2.w, pg.gC.x, fmaf(r3.x, pg.gC.y, fmaf(r3.y, pg.gC.z, ev.z * pg.gD)));
    // the pixel's state over the four pairs; the lane keeps its own w and ga
    float w = 0.f, ga = 0.f;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      if (!(hits & (0x11111111u << g))) continue;   // warp-uniform
      const float ag = __shfl_sync(0xffffffffu, ev.a, base | g);
      const float ig = __shfl_sync(0xffffffffu, iom, base | g);
      const float vg = __shfl_sync(0xffffffffu, vj, base | g);
      if (!((hits >> (base | g)) & 1u)) continue;
      const float Tb = st.T * ig;
      const float wg = ag * Tb;
      const float gg = Tb * vg - (st.acc - gOT) * ig;
      st.acc = fmaf(wg, vg, st.acc);
      st.T = Tb;
      if (e == g) {
        w = wg;
        ga = gg;
      }
    }
    __syncwarp();
    const float sv = ev.araw <= cfg.alpha_max ? -ev.G * r2.z * ga : 0.f;
    const float Px = fmaf(ev.u, r5.x, ev.v * r5.w);
    const float Py = fmaf(ev.u, r5.y, ev.v * r6.x);
    const float Pz = fmaf(ev.u, r5.z, ev.v * r6.y);
    const float Pr = fmaf(Px, rx, fmaf(Py, ry, Pz));
    const float beta = fmaf(sv, Pr, w * pg.gD) * fxfy * ev.rinv;
    const float Gx = fmaf(beta, r4.y, -sv * Px);
    const float Gy = fmaf(beta, r4.z, -sv * Py);
    const float Gz = fmaf(beta, r4.w, -sv * Pz);
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      if (!(hits & (0x11111111u << g))) continue;   // warp-uniform
      const float x = __shfl_sync(0xffffffffu, Gx, base | g);
      const float y = __shfl_sync(0xffffffffu, Gy, base | g);
      const float zc = __shfl_sync(0xffffffffu, Gz, base | g);
      const float z = __shfl_sync(0xffffffffu, ev.z, base | g);
      if (!((hits >> (base | g)) & 1u)) continue;
      st.sG.x += x;
      st.sG.y += y;
      st.sG.z += zc;
      st.szG.x = fmaf(z, x, st.szG.x);
      st.szG.y = fmaf(z, y, st.szG.y);
      st.szG.z = fmaf(z, zc, st.szG.z);
    }
    __syncwarp();
  }
}

}  // namespace gs2d
