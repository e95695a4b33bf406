// Map expansion (Sec. III-E): new surfels from a keyframe's RGB-D image,
// gated by a voxel hash table of the active map's occupied space.
//
// Passes (all on the caller's stream, no host round trip), one block per
// kExBlock = 1024 consecutive pixels in each:
//   select P_s     a bit per pixel (valid depth and u_keep < ratio) and the
//                  block's count;
//   points         per point of P_s, in pixel order: world position, the
//                  normal of Eq. normal_fromD from the observed depth, the
//                  create test (normal valid, voxel free), and the first
//                  P_s index of every 32-pixel word of the bit mask;
//   emit           per created point: the distance to its nearest other
//                  point of P_s (an exact windowed search in the image, see
//                  nearest_d2), then the surfel with its tangent frame,
//                  quaternion and state at n_map + rank; optionally its
//                  voxel is inserted into the table.
// A block's first index is the sum of the counts of the blocks before it,
// formed by the block itself (a scan launch more only beyond kSelfSumBlocks
// blocks, 4.2M pixels).
// Voxel table: open addressing with linear probing over 64-bit keys, every
// probe loop bounded by the capacity.
#include "gs2d_common.cuh"
#include "gs2d_expand.h"
#include "gs2d_internal.h"
#include "scan.cuh"

namespace gs2d {

constexpr int kExThreads = 256;
constexpr int kExPer = 4;                          // pixels per thread in the selection
constexpr int kExBlock = kExThreads * kExPer;
constexpr int kExWords = kExBlock / 32;            // mask words per block
constexpr unsigned long long kEmptyKey = ~0ull;
constexpr int kVoxBits = 21;
constexpr int kVoxHalf = 1 << (kVoxBits - 1);

__device__ __forceinline__ unsigned long long voxel_key(float x, float y, float z, float vox) {
  const float inv = 1.f / vox;
  int c[3] = {(int)floorf(x * inv), (int)floorf(y * inv), (int)floorf(z * inv)};
  unsigned long long k = 0ull;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int v = min(max(c[a], -kVoxHalf), kVoxHalf - 1) + kVoxHalf;
    k |= (unsigned long long)v << (kVoxBits * a);
  }
  return k;
}

// 64-bit finaliser of SplitMix64 (Steele, Lea, Flood 2014).
__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

__device__ __forceinline__ void voxel_put(const gs2d_voxel_table& t, unsigned long long key) {
  const uint32_t mask = t.capacity - 1u;
  uint32_t s = (uint32_t)mix64(key) & mask;
  for (uint32_t probe = 0; probe < t.capacity; ++probe, s = (s + 1u) & mask) {
    const unsigned long long prev = atomicCAS(reinterpret_cast<unsigned long long*>(t.keys) + s,
                                              kEmptyKey, key);
    if (prev == kEmptyKey || prev == key) return;
  }
  atomicExch(t.status, (int)GS2D_ERR_CAPACITY);
}

__device__ __forceinline__ bool voxel_has(const gs2d_voxel_table& t, unsigned long long key) {
  const uint32_t mask = t.capacity - 1u;
  uint32_t s = (uint32_t)mix64(key) & mask;
  for (uint32_t probe = 0; probe < t.capacity; ++probe, s = (s + 1u) & mask) {
    const unsigned long long k = t.keys[s];
    if (k == key) return true;
    if (k == kEmptyKey) return false;
  }
  return false;
}

__global__ void __launch_bounds__(kExThreads) voxel_clear_kernel(gs2d_voxel_table t) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < t.capacity;
       i += gridDim.x * blockDim.x)
    t.keys[i] = kEmptyKey;
  if (blockIdx.x == 0 && threadIdx.x == 0) *t.status = 0;
}

__global__ void __launch_bounds__(kExThreads) voxel_insert_kernel(gs2d_voxel_table t,
                                                                 const float* __restrict__ pts,
                                                                 const uint8_t* __restrict__ mask,
                                                                 int m) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    if (mask && !mask[i]) continue;
    voxel_put(t, voxel_key(pts[3 * i], pts[3 * i + 1], pts[3 * i + 2], t.voxel));
  }
}

__global__ void __launch_bounds__(kExThreads) voxel_query_kernel(gs2d_voxel_table t,
                                                                const float* __restrict__ pts,
                                                                int m, uint8_t* __restrict__ occ) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x)
    occ[i] = voxel_has(t, voxel_key(pts[3 * i], pts[3 * i + 1], pts[3 * i + 2], t.voxel)) ? 1 : 0;
}

// ---------------------------------------------------------------------------
// selection of P_s: a bit per pixel, counts per block of kExBlock pixels
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool depth_ok(float d) { return d > 0.f && d < INFINITY; }

__global__ void __launch_bounds__(kExThreads) ps_select_kernel(
    const float* __restrict__ depth, const float* __restrict__ u_keep, float ratio, int n,
    uint32_t* __restrict__ mask, int32_t* __restrict__ blk) {
  __shared__ int s_w[kExThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float d[kExPer], u[kExPer];
#pragma unroll
  for (int k = 0; k < kExPer; ++k) {   // word k * 8 + warp of the block
    const int p = blockIdx.x * kExBlock + k * kExThreads + (int)threadIdx.x;
    d[k] = p < n ? depth[p] : 0.f;
    u[k] = p < n ? u_keep[p] : 1.f;
  }
  int c = 0;
#pragma unroll
  for (int k = 0; k < kExPer; ++k) {
    const uint32_t b = __ballot_sync(0xffffffffu, depth_ok(d[k]) && u[k] < ratio);
    if (lane == 0) mask[blockIdx.x * kExWords + k * (kExThreads / 32) + warp] = b;
    c += __popc(b);
  }
  if (lane == 0) s_w[warp] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
#pragma unroll
    for (int w = 0; w < kExThreads / 32; ++w) t += s_w[w];
    blk[blockIdx.x] = t;
  }
}

// exclusive scan of nb block counts in place; *total = the sum (only for
// more than kSelfSumBlocks blocks)
__global__ void __launch_bounds__(kExThreads) select_scan_kernel(int32_t* __restrict__ blk, int nb,
                                                                int32_t* __restrict__ total) {
  __shared__ int s_w[kExThreads / 32];
  int carry = 0;
  for (int b0 = 0; b0 < nb; b0 += kExThreads) {
    const int b = b0 + (int)threadIdx.x;
    const int v = b < nb ? blk[b] : 0;
    int t;
    const int pre = block_exscan256(v, s_w, &t);
    if (b < nb) blk[b] = carry + pre;
    carry += t;
  }
  if (threadIdx.x == 0) *total = carry;
}

// ---------------------------------------------------------------------------
// points of P_s
// ---------------------------------------------------------------------------
__device__ __forceinline__ F3 back_project(const gs2d_camera& cam, int px, int py, float d) {
  return f3(d * ((px + 0.5f - cam.cx) / cam.fx), d * ((py + 0.5f - cam.cy) / cam.fy), d);
}

__device__ __forceinline__ F3 rot_t(const float* R, F3 v) {   // R^T v, R row-major
  return f3(R[0] * v.x + R[3] * v.y + R[6] * v.z, R[1] * v.x + R[4] * v.y + R[7] * v.z,
            R[2] * v.x + R[5] * v.y + R[8] * v.z);
}

// The points of the block's pixels, in pixel order at P_s indices base ..;
// word_at[w]: the P_s index of the first point of mask word w.
__global__ void __launch_bounds__(kExThreads) ps_point_kernel(
    const float* __restrict__ depth, gs2d_camera cam, const float* __restrict__ pose,
    const uint32_t* __restrict__ mask, const int32_t* __restrict__ blk, int nb,
    const int32_t* __restrict__ scanned_total, gs2d_voxel_table table, int use_table,
    int32_t* __restrict__ word_at, int32_t* __restrict__ idx, float4* __restrict__ pts,
    float4* __restrict__ nrm, uint8_t* __restrict__ create, int32_t* __restrict__ blk2) {
  __shared__ float T[12];   // T_cw: R row-major, t
  __shared__ int s_sum[16];
  __shared__ uint32_t s_mask[kExWords];
  __shared__ int s_at[kExWords + 1];
  __shared__ int s_p[kExBlock];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x < 12) T[threadIdx.x] = pose[threadIdx.x];
  int base, total;
  block_base(blk, nb, scanned_total, s_sum, &base, &total);
  if (warp == 0) {
    const uint32_t m = mask[blockIdx.x * kExWords + lane];
    int x = __popc(m);
    const int own = x;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, off);
      if (lane >= off) x += y;
    }
    s_mask[lane] = m;
    s_at[lane] = x - own;
    if (lane == 31) s_at[kExWords] = x;
    word_at[blockIdx.x * kExWords + lane] = base + x - own;
  }
  __syncthreads();
  const int cnt = s_at[kExWords];
  for (int w = warp; w < kExWords; w += kExThreads / 32) {
    const uint32_t m = s_mask[w];
    if ((m >> lane) & 1u)
      s_p[s_at[w] + __popc(m & ((1u << lane) - 1u))] = blockIdx.x * kExBlock + w * 32 + lane;
  }
  __syncthreads();
  const int W = cam.width, H = cam.height;
  int made = 0;
  for (int e = threadIdx.x; e < cnt; e += kExThreads) {
    const int k = base + e;
    const int p = s_p[e];
    const int px = p % W, py = p / W;
    const F3 Xc = back_project(cam, px, py, depth[p]);
    const F3 Xw = rot_t(T, f3(Xc.x - T[9], Xc.y - T[10], Xc.z - T[11]));
    idx[k] = p;
    pts[k] = make_float4(Xw.x, Xw.y, Xw.z, 0.f);
    // Eq. normal_fromD: central differences of the back-projected points
    bool ok = px >= 1 && py >= 1 && px < W - 1 && py < H - 1;
    F3 n = f3(0.f, 0.f, 0.f);
    if (ok) {
      const float dl = depth[p - 1], dr = depth[p + 1], du = depth[p - W], dd = depth[p + W];
      ok = depth_ok(dl) && depth_ok(dr) && depth_ok(du) && depth_ok(dd);
      if (ok) {
        const F3 xl = back_project(cam, px - 1, py, dl), xr = back_project(cam, px + 1, py, dr);
        const F3 xu = back_project(cam, px, py - 1, du), xd = back_project(cam, px, py + 1, dd);
        const F3 gx = 0.5f * (xr - xl), gy = 0.5f * (xd - xu);
        const F3 c = cross3(gx, gy);
        const float l2 = dot3(c, c);
        ok = l2 > 0.f;
        if (ok) n = rot_t(T, rsqrtf(l2) * c);
      }
    }
    bool free_vox = true;
    if (ok && use_table) free_vox = !voxel_has(table, voxel_key(Xw.x, Xw.y, Xw.z, table.voxel));
    nrm[k] = make_float4(n.x, n.y, n.z, sqrtf(dot3(Xc, Xc)));   // w: distance to the viewpoint
    create[k] = (ok && free_vox) ? 1 : 0;
    made += (ok && free_vox) ? 1 : 0;
  }
  made = __reduce_add_sync(0xffffffffu, made);
  __syncthreads();
  if (lane == 0) s_sum[warp] = made;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
#pragma unroll
    for (int w = 0; w < kExThreads / 32; ++w) t += s_sum[w];
    blk2[blockIdx.x] = t;
  }
}

// ---------------------------------------------------------------------------
// nearest other point of P_s
// ---------------------------------------------------------------------------
// P_s as the windowed search reads it.
struct PsGrid {
  const uint32_t* mask;     // a bit per pixel
  const int32_t* word_at;   // P_s index of each word's first point
  const float4* pts;
  int W, H;
  int m;                    // points in P_s
};

// Smallest squared distance (fmaf(dx, dx, fmaf(dy, dy, dz dz))) from q, the
// point j of pixel p, to the points of the mask words that meet the window
// of rx columns and ry rows about (px, py); a warp's lanes take the (row,
// word) pairs in turn.  A window of more pairs than P_s has points searches
// all of P_s instead (*all = true).
__device__ __forceinline__ float window_d2(const PsGrid& g, float4 q, int j, int p, int rx, int ry,
                                           int lane, bool* all) {
  const int px = p % g.W, py = p / g.W;
  const int x0 = max(px - rx, 0), x1 = min(px + rx, g.W - 1);
  const int y0 = max(py - ry, 0), y1 = min(py + ry, g.H - 1);
  // words a row's window can touch wherever it starts within a word
  const int nw = (x1 - x0) / 32 + 2, items = (y1 - y0 + 1) * nw;
  float best = INFINITY;
  auto take = [&](int k) {
    const float4 c = g.pts[k];
    const float ax = c.x - q.x, ay = c.y - q.y, az = c.z - q.z;
    best = fminf(best, fmaf(ax, ax, fmaf(ay, ay, az * az)));
  };
  *all = items >= g.m;
  if (*all) {
    for (int k = lane; k < g.m; k += 32)
      if (k != j) take(k);
  } else {
    for (int it = lane; it < items; it += 32) {
      const int r = it / nw;
      const int a = (y0 + r) * g.W + x0, b = a + (x1 - x0);   // the row's pixels a .. b
      const int w = (a >> 5) + (it - r * nw);
      if (w > (b >> 5)) continue;
      const uint32_t full = g.mask[w];
      uint32_t m = full;
      if (w == (p >> 5)) m &= ~(1u << (p & 31));              // the query itself
      if (!m) continue;
      const int at = g.word_at[w];
      while (m) {
        const int bit = __ffs(m) - 1;
        m &= m - 1u;
        take(at + __popc(full & ((1u << bit) - 1u)));
      }
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
    best = fminf(best, __shfl_xor_sync(0xffffffffu, best, off));
  return best;
}

// Columns (rows) on each side of pixel i that can hold a point within s of
// the query at depth d and ray coordinate x = (i + 0.5 - c) / f.  A point of
// column j lies on the plane through the eye and that column, at least
// d |x - x_j| / sqrt(1 + x_j^2) away; along j that distance has one maximum,
// so over the columns beyond r it is smallest at r + 1 or at the image edge.
// Infinite, NaN or huge s / d give the whole image.
__device__ __forceinline__ int reach(float s, float d, float c, float f, int i, int n) {
  const float x = (i + 0.5f - c) / f, step = 1.f / fabsf(f);
  const float xa = (0.5f - c) / f, xb = (n - 0.5f - c) / f;
  const float xm = fmaxf(fabsf(xa), fabsf(xb));
  const float t = s / d;
  const float loose = t * sqrtf(fmaf(xm, xm, 1.f)) / step;
  if (!(loose < (float)n)) return n;
  const int r_loose = (int)loose + 1;
  // tighter: the bound of the columns just outside the loose window
  const float xl = fabsf(x) + (r_loose + 1) * step;
  const int r = (int)(t * sqrtf(fmaf(xl, xl, 1.f)) / step) + 1;
  const bool edges = fabsf(x - xa) >= t * sqrtf(fmaf(xa, xa, 1.f)) &&
                     fabsf(x - xb) >= t * sqrtf(fmaf(xb, xb, 1.f));
  return (edges && r < r_loose) ? r : r_loose;
}

// Squared distance from the point k of pixel p to its nearest other point
// of P_s (INFINITY if there is none): exactly the minimum over all of them.
// A window that grows until it holds a point gives an upper bound s; the
// points within s all lie in the window that `reach` derives from it, and
// that window is searched.  bound_scale and bound_abs make the window cover
// the rounding of the 32-bit points and an R that is not quite a rotation
// (its smallest singular value is at least bound_scale).
// One warp per query; the work per query is that of its window (~20 mask
// words, ~10 points) or at most that of all points, where an exhaustive
// search staged all of them for every query: 32k points of a 1200x680
// keyframe, 349 us -> 18 us for the whole emit kernel, which is bound by the
// latency of its dependent reads (mask, index, point; all in L2).
__device__ __forceinline__ float nearest_d2(const PsGrid& g, const gs2d_camera& cam, int j, int p,
                                            float d, float bound_scale, float bound_abs, int r0,
                                            int lane) {
  const float4 q = g.pts[j];
  float best = INFINITY;
  int r = r0;
  bool all = false;
  while (true) {
    best = window_d2(g, q, j, p, r, r, lane, &all);
    if (all || best < INFINITY || r >= max(g.W, g.H)) break;
    r = min(2 * r, max(g.W, g.H));
  }
  if (all || !(best < INFINITY)) return best;
  const float s = (sqrtf(best) * 1.0001f + bound_abs) / bound_scale;
  const int rx = reach(s, d, cam.cx, cam.fx, p % g.W, g.W);
  const int ry = reach(s, d, cam.cy, cam.fy, p / g.W, g.H);
  if (rx <= r && ry <= r) return best;
  return fminf(best, window_d2(g, q, j, p, rx, ry, lane, &all));
}

struct EmitArgs {
  const float* rgb;
  const float* depth;
  const float* u_angle;
  const float* pose;
  gs2d_camera cam;
  PsGrid g;
  const int32_t* idx;      // pixel of each P_s point
  const float4* nrm;
  const uint8_t* create;
  float max_scale;
  const int32_t* blk2;     // created points per block (exclusive sums when scanned)
  int nb;
  const int32_t* scanned_total;
  float* mu;
  float* quat;
  float* scale;
  float* opacity;
  float* rgb_out;
  gs2d_map_state st;
  int n_map, capacity;
  float opac0;
  int kf_id;
  gs2d_voxel_table table;
  int insert;
  int32_t* n_new;
};

__device__ __forceinline__ void emit_one(const EmitArgs& a, int j, float d2, int o) {
  const int p = a.idx[j];
  const float4 X = a.g.pts[j];
  const float4 N = a.nrm[j];
  // orthonormal basis of the normal's plane (Duff et al. 2017)
  const float sg = copysignf(1.f, N.z);
  const float aa = -1.f / (sg + N.z);
  const float bb = N.x * N.y * aa;
  const F3 b1 = f3(1.f + sg * N.x * N.x * aa, sg * bb, -sg * N.x);
  const F3 b2 = f3(bb, sg + N.y * N.y * aa, -N.y);
  float sp, cp;
  sincospif(2.f * a.u_angle[p], &sp, &cp);
  const F3 tn = f3(N.x, N.y, N.z);
  const F3 tu = cp * b1 + sp * b2;
  const F3 tv = cross3(tn, tu);
  const float D[9] = {tu.x, tv.x, tn.x, tu.y, tv.y, tn.y, tu.z, tv.z, tn.z};
  a.mu[3 * o] = X.x;
  a.mu[3 * o + 1] = X.y;
  a.mu[3 * o + 2] = X.z;
  reinterpret_cast<float4*>(a.quat)[o] = quat_from_matrix(D);
  const float s = d2 < INFINITY ? sqrtf(d2) : a.max_scale;
  a.scale[2 * o] = s;
  a.scale[2 * o + 1] = s;
  a.opacity[o] = a.opac0;
  a.rgb_out[3 * o] = a.rgb[3 * p];
  a.rgb_out[3 * o + 1] = a.rgb[3 * p + 1];
  a.rgb_out[3 * o + 2] = a.rgb[3 * p + 2];
  if (a.st.delta) a.st.delta[o] = 1;
  if (a.st.t_c) a.st.t_c[o] = a.kf_id;
  if (a.st.t_l) a.st.t_l[o] = a.kf_id;
  if (a.st.d_c) a.st.d_c[o] = N.w;
  if (a.insert) voxel_put(a.table, voxel_key(X.x, X.y, X.z, a.table.voxel));
}

// The block's created points, in pixel order: first a warp per point finds
// its nearest neighbour, then a thread per point writes the surfel.
__global__ void __launch_bounds__(kExThreads) emit_kernel(EmitArgs a) {
  __shared__ int s_sum[16];
  __shared__ int s_w[kExThreads / 32];
  __shared__ int s_j[kExBlock];
  __shared__ float s_d2[kExBlock];
  __shared__ float s_bound[2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int first, total;
  block_base(a.blk2, a.nb, a.scanned_total, s_sum, &first, &total);
  const bool fits = (long long)a.n_map + total <= a.capacity;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *a.n_new = total;
    if (!fits && a.table.status) atomicExch(a.table.status, (int)GS2D_ERR_CAPACITY);
  }
  if (!fits) return;
  // the block's points of P_s: word_at of its first word .. past its last
  const int w0 = blockIdx.x * kExWords, wl = a.nb * kExWords - 1;
  a.g.m = a.g.word_at[wl] + __popc(a.g.mask[wl]);
  const int lo = a.g.word_at[w0];
  const int hi = a.g.word_at[w0 + kExWords - 1] + __popc(a.g.mask[w0 + kExWords - 1]);
  int made = 0;
  for (int e0 = lo; e0 < hi; e0 += kExThreads) {
    const int j = e0 + (int)threadIdx.x;
    const int f = (j < hi && a.create[j]) ? 1 : 0;
    int t;
    const int o = made + block_exscan256(f, s_w, &t);
    if (f) s_j[o] = j;
    made += t;
  }
  if (threadIdx.x == 0) {
    // R^T R = I + E: every singular value of R is at least sqrt(1 - |E|_F)
    const float* R = a.pose;
    float e2 = 0.f;
    for (int r = 0; r < 3; ++r)
      for (int c = 0; c < 3; ++c) {
        const float v = R[3 * r] * R[3 * c] + R[3 * r + 1] * R[3 * c + 1] +
                        R[3 * r + 2] * R[3 * c + 2] - (r == c ? 1.f : 0.f);
        e2 = fmaf(v, v, e2);
      }
    s_bound[0] = sqrtf(fmaxf(1.f - sqrtf(e2) - 1e-6f, 0.f));
    s_bound[1] = fabsf(R[9]) + fabsf(R[10]) + fabsf(R[11]);
  }
  __syncthreads();
  // first window: about nine points on average
  const int r0 = max(1, (int)(1.5f * sqrtf((float)kExBlock / (float)max(hi - lo, 1))));
  for (int e = warp; e < made; e += kExThreads / 32) {
    const int j = s_j[e];
    const int p = a.idx[j];
    // 16 units of rounding at the scale of the points' coordinates
    const float abs_err = 2e-6f * (a.nrm[j].w + s_bound[1]) * 8.f;
    const float d2 = nearest_d2(a.g, a.cam, j, p, a.depth[p], s_bound[0], abs_err, r0, lane);
    if (lane == 0) s_d2[e] = d2;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < made; e += kExThreads) emit_one(a, s_j[e], s_d2[e], a.n_map + first + e);
}

struct ExWs {
  int32_t *blk, *blk2, *m, *k, *word_at, *idx;
  uint32_t* mask;
  float4 *pts, *nrm;
  uint8_t* create;
  size_t bytes;
};

ExWs carve_expand(void* base, int P) {
  Carver c(base);
  ExWs w;
  const int nb = (P + kExBlock - 1) / kExBlock;
  w.blk = c.take<int32_t>(nb);
  w.blk2 = c.take<int32_t>(nb);
  w.m = c.take<int32_t>(1);
  w.k = c.take<int32_t>(1);
  w.mask = c.take<uint32_t>((size_t)nb * kExWords);
  w.word_at = c.take<int32_t>((size_t)nb * kExWords);
  w.idx = c.take<int32_t>(P);
  w.pts = c.take<float4>(P);
  w.nrm = c.take<float4>(P);
  w.create = c.take<uint8_t>(P);
  w.bytes = align_up(c.off, 256);
  return w;
}

bool table_ok(const gs2d_voxel_table* t) {
  return t && t->keys && t->status && t->capacity > 0 && (t->capacity & (t->capacity - 1)) == 0 &&
         t->voxel > 0.f;
}

int blocks_for(long long n) { return (int)max(1ll, min((n + kExThreads - 1) / kExThreads, 152ll * 32)); }

}  // namespace gs2d

using namespace gs2d;

extern "C" {

int gs2d_voxel_clear(const gs2d_voxel_table* t, gs2d_stream stream) {
  if (!table_ok(t)) return GS2D_ERR_INVALID_ARG;
  voxel_clear_kernel<<<blocks_for(t->capacity), kExThreads, 0, (cudaStream_t)stream>>>(*t);
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

int gs2d_voxel_insert(const gs2d_voxel_table* t, const float* points, const uint8_t* mask, int m,
                      gs2d_stream stream) {
  if (!table_ok(t) || m < 0 || (m > 0 && !points)) return GS2D_ERR_INVALID_ARG;
  if (m == 0) return GS2D_OK;
  voxel_insert_kernel<<<blocks_for(m), kExThreads, 0, (cudaStream_t)stream>>>(*t, points, mask, m);
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

int gs2d_voxel_query(const gs2d_voxel_table* t, const float* points, int m, uint8_t* occupied,
                     gs2d_stream stream) {
  if (!table_ok(t) || m < 0 || (m > 0 && (!points || !occupied))) return GS2D_ERR_INVALID_ARG;
  if (m == 0) return GS2D_OK;
  voxel_query_kernel<<<blocks_for(m), kExThreads, 0, (cudaStream_t)stream>>>(*t, points, m,
                                                                           occupied);
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

size_t gs2d_expand_workspace(const gs2d_camera* cam) {
  if (!cam || cam->width <= 0 || cam->height <= 0) return 0;
  return carve_expand(nullptr, cam->width * cam->height).bytes;
}

int gs2d_expand(const float* rgb, const float* depth, const gs2d_camera* cam, const float* pose_cw,
                const float* u_keep, const float* u_angle, const gs2d_voxel_table* table,
                const gs2d_expand_params* prm, int n_map, int capacity, float* mu, float* quat,
                float* scale, float* opacity, float* rgb_out, const gs2d_map_state* st,
                int32_t* n_new, void* workspace, size_t ws_bytes, size_t* ws_needed,
                gs2d_stream stream) {
  if (!cam || cam->width <= 0 || cam->height <= 0 || !prm || !n_new) return GS2D_ERR_INVALID_ARG;
  if ((long long)cam->width * cam->height > (1ll << 30)) return GS2D_ERR_INVALID_ARG;
  const int P = cam->width * cam->height;
  const ExWs sz = carve_expand(nullptr, P);
  if (ws_needed) *ws_needed = sz.bytes;
  if (!workspace || ws_bytes < sz.bytes) return GS2D_ERR_WORKSPACE;
  if (!rgb || !depth || !pose_cw || !u_keep || !u_angle || !mu || !quat || !scale || !opacity ||
      !rgb_out || n_map < 0 || capacity < n_map || !(prm->ratio > 0.f && prm->ratio <= 1.f))
    return GS2D_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(quat) & 15) return GS2D_ERR_INVALID_ARG;
  if (table && !table_ok(table)) return GS2D_ERR_INVALID_ARG;
  if (prm->insert_new && !table) return GS2D_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  const ExWs w = carve_expand(workspace, P);
  const int nb = (P + kExBlock - 1) / kExBlock;
  const bool scan = nb > kSelfSumBlocks;
  ps_select_kernel<<<nb, kExThreads, 0, s>>>(depth, u_keep, prm->ratio, P, w.mask, w.blk);
  GS2D_LAUNCH_CHECK();
  if (scan) {
    select_scan_kernel<<<1, kExThreads, 0, s>>>(w.blk, nb, w.m);
    GS2D_LAUNCH_CHECK();
  }
  const gs2d_voxel_table tb = table ? *table : gs2d_voxel_table{nullptr, 0u, 1.f, nullptr};
  ps_point_kernel<<<nb, kExThreads, 0, s>>>(depth, *cam, pose_cw, w.mask, w.blk, nb,
                                            scan ? w.m : nullptr, tb, table ? 1 : 0, w.word_at,
                                            w.idx, w.pts, w.nrm, w.create, w.blk2);
  GS2D_LAUNCH_CHECK();
  if (scan) {
    select_scan_kernel<<<1, kExThreads, 0, s>>>(w.blk2, nb, w.k);
    GS2D_LAUNCH_CHECK();
  }
  EmitArgs a;
  a.rgb = rgb;
  a.depth = depth;
  a.u_angle = u_angle;
  a.pose = pose_cw;
  a.cam = *cam;
  a.g = PsGrid{w.mask, w.word_at, w.pts, cam->width, cam->height, 0};
  a.idx = w.idx;
  a.nrm = w.nrm;
  a.create = w.create;
  a.max_scale = prm->max_scale;
  a.blk2 = w.blk2;
  a.nb = nb;
  a.scanned_total = scan ? w.k : nullptr;
  a.mu = mu;
  a.quat = quat;
  a.scale = scale;
  a.opacity = opacity;
  a.rgb_out = rgb_out;
  a.st = st ? *st : gs2d_map_state{nullptr, nullptr, nullptr, nullptr};
  a.n_map = n_map;
  a.capacity = capacity;
  a.opac0 = prm->opacity;
  a.kf_id = prm->kf_id;
  a.table = tb;
  a.insert = prm->insert_new;
  a.n_new = n_new;
  emit_kernel<<<nb, kExThreads, 0, s>>>(a);
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

}  // extern "C"
