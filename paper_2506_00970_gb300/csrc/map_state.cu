// Map state of 2DGS-SLAM (Eq. map): the per-keyframe state update of
// Sec. III-F, the map correction of Sec. IV-C, the occlusion pruning of
// Sec. III-F and a stable compaction of the surfel arrays.  All of them are
// one pass over the map's structure-of-arrays, loads and stores coalesced per
// array, a thread's four items in flight together; bound by HBM.
#include "gs2d_common.cuh"
#include "gs2d_internal.h"
#include "gs2d_map.h"
#include "scan.cuh"

namespace gs2d {

constexpr int kMapThreads = 256;
constexpr int kMapMaxBlocks = 152 * 32;
constexpr int kMapPer = 4;                             // items per thread
constexpr int kCompactPer = 4;                         // items per thread
constexpr int kCompactBlock = kMapThreads * kCompactPer;

__host__ __device__ inline int map_blocks(int n) {
  const int b = (n + kMapThreads - 1) / kMapThreads;
  return b < 1 ? 1 : (b > kMapMaxBlocks ? kMapMaxBlocks : b);
}

__host__ __device__ inline int map_blocks4(int n) {
  return map_blocks((n + kMapPer - 1) / kMapPer);
}

// Adds a block's sum of c to *counter, one atomic per block.  s: 8 ints.
__device__ __forceinline__ void block_count_add(int c, int* s, uint32_t* counter) {
  c = __reduce_add_sync(0xffffffffu, c);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
#pragma unroll
    for (int w = 0; w < kMapThreads / 32; ++w) t += s[w];
    if (t) atomicAdd(counter, (uint32_t)t);
  }
}

// Block b takes items b * 1024 + k * 256 + thread, k < 4.  One counter atomic
// per block (one per warp and counter serialised on four addresses): 2M
// surfels 48 -> 18 us.
__global__ void __launch_bounds__(kMapThreads) map_observe_kernel(
    const float* __restrict__ contrib, const float* __restrict__ mu, int n,
    const float* __restrict__ pose, int kf, gs2d_state_params prm, gs2d_map_state st,
    uint32_t* __restrict__ counts) {
  __shared__ int s_w[kMapThreads / 32];
  // camera centre c = -R^T t of the keyframe
  const float cx = -(pose[0] * pose[9] + pose[3] * pose[10] + pose[6] * pose[11]);
  const float cy = -(pose[1] * pose[9] + pose[4] * pose[10] + pose[7] * pose[11]);
  const float cz = -(pose[2] * pose[9] + pose[5] * pose[10] + pose[8] * pose[11]);
  int vis_act = 0, closer = 0, deact = 0, react = 0;
  for (long long b = blockIdx.x; b * (kMapThreads * kMapPer) < n; b += gridDim.x) {
    const int base = (int)b * (kMapThreads * kMapPer) + (int)threadIdx.x;
    bool vis[kMapPer];
    uint8_t act[kMapPer];
    int tl[kMapPer];
#pragma unroll
    for (int k = 0; k < kMapPer; ++k) {
      const int i = base + k * kMapThreads;
      const bool in = i < n;
      vis[k] = in && contrib[i] > prm.vis_threshold;
      act[k] = in ? st.delta[i] : 0;
      tl[k] = in ? st.t_l[i] : kf;
    }
    float d[kMapPer], dc[kMapPer];
#pragma unroll
    for (int k = 0; k < kMapPer; ++k) {
      const int i = base + k * kMapThreads;
      d[k] = dc[k] = 0.f;
      if (vis[k] && act[k]) {
        const float dx = mu[3 * (size_t)i] - cx, dy = mu[3 * (size_t)i + 1] - cy,
                    dz = mu[3 * (size_t)i + 2] - cz;
        d[k] = sqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
        dc[k] = st.d_c[i];
      }
    }
#pragma unroll
    for (int k = 0; k < kMapPer; ++k) {
      const int i = base + k * kMapThreads;
      if (i >= n) continue;
      if (act[k]) {
        int t = tl[k];
        if (vis[k]) {
          ++vis_act;
          t = kf;
          st.t_l[i] = kf;
          if (d[k] < dc[k]) {
            st.d_c[i] = d[k];
            st.t_c[i] = kf;
            ++closer;
          }
        }
        if ((long long)kf - t > prm.inactive_after) {
          st.delta[i] = 0;
          ++deact;
        }
      } else if (prm.reactivate && vis[k] && st.t_c[i] > prm.loop_h) {
        st.delta[i] = 1;
        st.t_l[i] = kf;
        ++react;
      }
    }
  }
  if (counts) {
    block_count_add(vis_act, s_w, counts);
    block_count_add(closer, s_w, counts + 1);
    block_count_add(deact, s_w, counts + 2);
    block_count_add(react, s_w, counts + 3);
  }
}

// Pose increments dT_j = (T^o_cw)^-1 T_cw: dR = R_o^T R, dt = R_o^T (t - t_o),
// and the unit quaternion of dR.
// Record layout: dR [9], dt [3], q [4] (w, x, y, z).
__global__ void map_delta_kernel(const float* __restrict__ old_p, const float* __restrict__ new_p,
                                 int n_kf, float* __restrict__ delta) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n_kf) return;
  const float* A = old_p + 12 * j;
  const float* B = new_p + 12 * j;
  float D[9], t[3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
      D[3 * r + c] = B[r] * A[c] + B[3 + r] * A[3 + c] + B[6 + r] * A[6 + c];
    t[r] = B[r] * (A[9] - B[9]) + B[3 + r] * (A[10] - B[10]) + B[6 + r] * (A[11] - B[11]);
  }
  const float4 q = quat_from_matrix(D);
  float* o = delta + 16 * j;
#pragma unroll
  for (int k = 0; k < 9; ++k) o[k] = D[k];
  o[9] = t[0];
  o[10] = t[1];
  o[11] = t[2];
  o[12] = q.x;
  o[13] = q.y;
  o[14] = q.z;
  o[15] = q.w;
}

// The increments are gathered by every surfel: up to kSharedKf of them are
// staged in shared memory, rows padded to 20 floats (a warp's 16-byte reads
// of random rows then spread over the banks), in place of 16 scalar gathers
// from L1, and skipped surfels are counted once per block; 2M surfels, 64
// keyframes: 53 -> 20 us.
constexpr int kSharedKf = 512;   // 40 KB
template <bool kShared>
__global__ void __launch_bounds__(kMapThreads) map_correct_kernel(
    float* __restrict__ mu, float4* __restrict__ quat, const int32_t* __restrict__ t_c, int n,
    const float* __restrict__ delta, int n_kf, int32_t* __restrict__ n_skipped) {
  extern __shared__ float4 s_delta[];   // [n_kf][5]
  __shared__ int s_w[kMapThreads / 32];
  if (kShared) {
    float* s = reinterpret_cast<float*>(s_delta);
    for (int e = threadIdx.x; e < 16 * n_kf; e += kMapThreads)
      s[(e >> 4) * 20 + (e & 15)] = delta[e];
    __syncthreads();
  }
  int skipped = 0;
  for (long long b = blockIdx.x; b * (kMapThreads * kMapPer) < n; b += gridDim.x) {
    const int base = (int)b * (kMapThreads * kMapPer) + (int)threadIdx.x;
    int j[kMapPer];
    float x[kMapPer], y[kMapPer], z[kMapPer];
    float4 q[kMapPer];
#pragma unroll
    for (int k = 0; k < kMapPer; ++k) {
      const int i = base + k * kMapThreads;
      j[k] = -1;
      if (i < n) {
        j[k] = t_c[i];
        x[k] = mu[3 * (size_t)i];
        y[k] = mu[3 * (size_t)i + 1];
        z[k] = mu[3 * (size_t)i + 2];
        q[k] = quat[i];                             // (w, x, y, z)
        if (j[k] < 0 || j[k] >= n_kf) {
          j[k] = -1;
          ++skipped;
        }
      }
    }
#pragma unroll
    for (int k = 0; k < kMapPer; ++k) {
      if (j[k] < 0) continue;
      const int i = base + k * kMapThreads;
      float d[16];
      if (kShared) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float4 v = s_delta[j[k] * 5 + c];
          d[4 * c] = v.x;
          d[4 * c + 1] = v.y;
          d[4 * c + 2] = v.z;
          d[4 * c + 3] = v.w;
        }
      } else {
#pragma unroll
        for (int c = 0; c < 16; ++c) d[c] = delta[16 * (size_t)j[k] + c];
      }
      mu[3 * (size_t)i] = fmaf(d[0], x[k], fmaf(d[1], y[k], fmaf(d[2], z[k], d[9])));
      mu[3 * (size_t)i + 1] = fmaf(d[3], x[k], fmaf(d[4], y[k], fmaf(d[5], z[k], d[10])));
      mu[3 * (size_t)i + 2] = fmaf(d[6], x[k], fmaf(d[7], y[k], fmaf(d[8], z[k], d[11])));
      const float aw = d[12], ax = d[13], ay = d[14], az = d[15];
      // Hamilton product q(dR) q: R(q(dR) q) = dR R(q)
      quat[i] = make_float4(aw * q[k].x - ax * q[k].y - ay * q[k].z - az * q[k].w,
                            aw * q[k].y + ax * q[k].x + ay * q[k].w - az * q[k].z,
                            aw * q[k].z - ax * q[k].w + ay * q[k].x + az * q[k].y,
                            aw * q[k].w + ax * q[k].z - ay * q[k].y + az * q[k].x);
    }
  }
  if (n_skipped) block_count_add(skipped, s_w, reinterpret_cast<uint32_t*>(n_skipped));
}

__global__ void __launch_bounds__(kMapThreads) map_prune_kernel(const float* __restrict__ contrib,
                                                                const int32_t* __restrict__ t_c,
                                                                int n, int r, float thr,
                                                                uint8_t* __restrict__ keep) {
  for (long long b = blockIdx.x; b * (kMapThreads * kMapPer) < n; b += gridDim.x) {
    const int base = (int)b * (kMapThreads * kMapPer) + (int)threadIdx.x;
    bool out[kMapPer];
#pragma unroll
    for (int k = 0; k < kMapPer; ++k) {
      const int i = base + k * kMapThreads;
      out[k] = i < n && t_c[i] == r && contrib[i] < thr;
    }
#pragma unroll
    for (int k = 0; k < kMapPer; ++k)
      if (base + k * kMapThreads < n) keep[base + k * kMapThreads] = out[k] ? 0 : 1;
  }
}

// Compaction, pass 1: kept items per block of kCompactBlock (item
// base + k * 256 + thread for k < 4: each warp access is 32 consecutive items).
__global__ void __launch_bounds__(kMapThreads) compact_count_kernel(const uint8_t* __restrict__ keep,
                                                                    int n,
                                                                    int32_t* __restrict__ blk) {
  __shared__ int s_w[kMapThreads / 32];
  const int base = blockIdx.x * kCompactBlock + threadIdx.x;
  int c = 0;
#pragma unroll
  for (int k = 0; k < kCompactPer; ++k) {
    const int i = base + k * kMapThreads;
    c += (i < n && keep[i]) ? 1 : 0;
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) c += __shfl_xor_sync(0xffffffffu, c, off);
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int s = 0;
    for (int w = 0; w < kMapThreads / 32; ++w) s += s_w[w];
    blk[blockIdx.x] = s;
  }
}

// For more than kSelfSumBlocks blocks: exclusive scan of the block counts, in
// place; *n_out = the total.
__global__ void __launch_bounds__(kMapThreads) compact_scan_kernel(int32_t* __restrict__ blk,
                                                                   int nb,
                                                                   int32_t* __restrict__ n_out) {
  __shared__ int s_w[kMapThreads / 32];
  int carry = 0;
  for (int b0 = 0; b0 < nb; b0 += kMapThreads) {
    const int b = b0 + (int)threadIdx.x;
    const int v = b < nb ? blk[b] : 0;
    int total;
    const int pre = block_exscan256(v, s_w, &total);
    if (b < nb) blk[b] = carry + pre;
    carry += total;
  }
  if (threadIdx.x == 0) *n_out = carry;
}

template <int W, typename T>
__device__ __forceinline__ void copy_kept(const T* __restrict__ in, T* __restrict__ out,
                                          const int (&src)[kCompactPer],
                                          const int (&dst)[kCompactPer]) {
  T v[kCompactPer][W];
#pragma unroll
  for (int k = 0; k < kCompactPer; ++k)
#pragma unroll
    for (int c = 0; c < W; ++c)
      if (dst[k] >= 0) v[k][c] = in[(size_t)src[k] * W + c];
#pragma unroll
  for (int k = 0; k < kCompactPer; ++k)
#pragma unroll
    for (int c = 0; c < W; ++c)
      if (dst[k] >= 0) out[(size_t)dst[k] * W + c] = v[k][c];
}

// Pass 2: every kept item to its slot.  The block ranks its four runs of 256
// consecutive items at once (two barriers), then copies array by array, a
// thread's four items in flight together (coalesced loads and, for runs of
// kept items, coalesced stores): 2M surfels 59 -> 54 us, 5.0 TB/s of the 272 MB moved, and
// no scan launch (7.8 us) before it.
__global__ void __launch_bounds__(kMapThreads) compact_scatter_kernel(
    const uint8_t* __restrict__ keep, int n, const int32_t* __restrict__ blk, int nb,
    int32_t* __restrict__ n_out, int scanned, gs2d_surfels s,
    gs2d_map_state st, float* __restrict__ mu_o, float* __restrict__ quat_o,
    float* __restrict__ scale_o, float* __restrict__ opac_o, float* __restrict__ rgb_o,
    gs2d_map_state so, int32_t* __restrict__ new_index) {
  __shared__ int s_sum[16];
  __shared__ int s_c[kCompactPer * (kMapThreads / 32)];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int src[kCompactPer], dst[kCompactPer];
  uint32_t bal[kCompactPer];
#pragma unroll
  for (int k = 0; k < kCompactPer; ++k) {
    src[k] = blockIdx.x * kCompactBlock + k * kMapThreads + (int)threadIdx.x;
    bal[k] = __ballot_sync(0xffffffffu, src[k] < n && keep[src[k]]);
    if (lane == 0) s_c[k * (kMapThreads / 32) + warp] = __popc(bal[k]);
  }
  int carry, total;
  block_base(blk, nb, scanned ? n_out : nullptr, s_sum, &carry, &total);
  if (scanned) __syncthreads();
  if (!scanned && blockIdx.x == 0 && threadIdx.x == 0) *n_out = total;
#pragma unroll
  for (int k = 0; k < kCompactPer; ++k) {
    int o = carry + __popc(bal[k] & ((1u << lane) - 1u));
#pragma unroll
    for (int w = 0; w < kMapThreads / 32; ++w) {
      const int c = s_c[k * (kMapThreads / 32) + w];
      if (w < warp) o += c;
      carry += c;
    }
    dst[k] = (bal[k] >> lane) & 1u ? o : -1;
    if (src[k] < n && new_index) new_index[src[k]] = dst[k];
  }
  copy_kept<3>(s.mu, mu_o, src, dst);
  copy_kept<1>(reinterpret_cast<const float4*>(s.quat), reinterpret_cast<float4*>(quat_o), src, dst);
  copy_kept<2>(s.scale, scale_o, src, dst);
  copy_kept<1>(s.opacity, opac_o, src, dst);
  copy_kept<3>(s.rgb, rgb_o, src, dst);
  if (st.delta) copy_kept<1>(st.delta, so.delta, src, dst);
  if (st.t_c) copy_kept<1>(st.t_c, so.t_c, src, dst);
  if (st.d_c) copy_kept<1>(st.d_c, so.d_c, src, dst);
  if (st.t_l) copy_kept<1>(st.t_l, so.t_l, src, dst);
}

__global__ void __launch_bounds__(kMapThreads) map_expand_values_kernel(
    const float* __restrict__ vals, const int32_t* __restrict__ idx, int n, float fill,
    float* __restrict__ out) {
  const int stride = gridDim.x * blockDim.x;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const int k = idx[i];
    out[i] = k >= 0 ? vals[k] : fill;
  }
}

}  // namespace gs2d

using namespace gs2d;

extern "C" {

int gs2d_map_observe(const float* contrib, const float* mu, int n, const float* pose_cw,
                     int kf_id, const gs2d_state_params* prm, const gs2d_map_state* st,
                     uint32_t* counts, gs2d_stream stream) {
  if (n < 0 || !prm || !st || !pose_cw) return GS2D_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  if (counts && cudaMemsetAsync(counts, 0, 4 * sizeof(uint32_t), s) != cudaSuccess)
    return GS2D_ERR_CUDA;
  if (n == 0) return GS2D_OK;
  if (!contrib || !mu || !st->delta || !st->t_c || !st->d_c || !st->t_l)
    return GS2D_ERR_INVALID_ARG;
  map_observe_kernel<<<map_blocks4(n), kMapThreads, 0, s>>>(contrib, mu, n, pose_cw, kf_id, *prm,
                                                           *st, counts);
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

size_t gs2d_map_correct_workspace(int n_kf) {
  return align_up((size_t)(n_kf > 0 ? n_kf : 1) * 16 * sizeof(float), 256);
}

int gs2d_map_correct(float* mu, float* quat, const int32_t* t_c, int n, const float* poses_old,
                     const float* poses_new, int n_kf, void* workspace, size_t ws_bytes,
                     size_t* ws_needed, int32_t* n_skipped, gs2d_stream stream) {
  if (n < 0 || n_kf < 0) return GS2D_ERR_INVALID_ARG;
  const size_t need = gs2d_map_correct_workspace(n_kf);
  if (ws_needed) *ws_needed = need;
  if (!workspace || ws_bytes < need) return GS2D_ERR_WORKSPACE;
  cudaStream_t s = (cudaStream_t)stream;
  if (n_skipped && cudaMemsetAsync(n_skipped, 0, sizeof(int32_t), s) != cudaSuccess)
    return GS2D_ERR_CUDA;
  if (n == 0) return GS2D_OK;
  if (!mu || !quat || !t_c || (n_kf > 0 && (!poses_old || !poses_new)))
    return GS2D_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(quat) & 15) return GS2D_ERR_INVALID_ARG;
  float* delta = static_cast<float*>(workspace);
  if (n_kf > 0) {
    map_delta_kernel<<<(n_kf + 127) / 128, 128, 0, s>>>(poses_old, poses_new, n_kf, delta);
    GS2D_LAUNCH_CHECK();
  }
  float4* q4 = reinterpret_cast<float4*>(quat);
  if (n_kf <= kSharedKf)
    map_correct_kernel<true><<<map_blocks4(n), kMapThreads, (size_t)n_kf * 5 * sizeof(float4), s>>>(
        mu, q4, t_c, n, delta, n_kf, n_skipped);
  else
    map_correct_kernel<false><<<map_blocks4(n), kMapThreads, 0, s>>>(mu, q4, t_c, n, delta, n_kf,
                                                                     n_skipped);
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

int gs2d_map_prune(const float* contrib, const int32_t* t_c, int n, int r, float vis_threshold,
                   uint8_t* keep, gs2d_stream stream) {
  if (n < 0) return GS2D_ERR_INVALID_ARG;
  if (n == 0) return GS2D_OK;
  if (!contrib || !t_c || !keep) return GS2D_ERR_INVALID_ARG;
  map_prune_kernel<<<map_blocks4(n), kMapThreads, 0, (cudaStream_t)stream>>>(contrib, t_c, n, r,
                                                                           vis_threshold, keep);
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

int gs2d_map_expand_values(const float* vals, const int32_t* new_index, int n, float fill,
                           float* out, gs2d_stream stream) {
  if (n < 0) return GS2D_ERR_INVALID_ARG;
  if (n == 0) return GS2D_OK;
  if (!vals || !new_index || !out) return GS2D_ERR_INVALID_ARG;
  map_expand_values_kernel<<<map_blocks(n), kMapThreads, 0, (cudaStream_t)stream>>>(
      vals, new_index, n, fill, out);
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

size_t gs2d_map_compact_workspace(int n) {
  const size_t nb = (size_t)((n > 0 ? n : 1) + kCompactBlock - 1) / kCompactBlock;
  return align_up(nb * sizeof(int32_t), 256);
}

int gs2d_map_compact(const uint8_t* keep, int n, const gs2d_surfels* s, const gs2d_map_state* st,
                     float* mu_out, float* quat_out, float* scale_out, float* opacity_out,
                     float* rgb_out, const gs2d_map_state* st_out, int32_t* new_index,
                     int32_t* n_out, void* workspace, size_t ws_bytes, size_t* ws_needed,
                     gs2d_stream stream) {
  if (n < 0 || !s || !n_out) return GS2D_ERR_INVALID_ARG;
  const size_t need = gs2d_map_compact_workspace(n);
  if (ws_needed) *ws_needed = need;
  if (!workspace || ws_bytes < need) return GS2D_ERR_WORKSPACE;
  cudaStream_t cs = (cudaStream_t)stream;
  if (n == 0) {
    if (cudaMemsetAsync(n_out, 0, sizeof(int32_t), cs) != cudaSuccess) return GS2D_ERR_CUDA;
    return GS2D_OK;
  }
  if (!keep || !s->mu || !s->quat || !s->scale || !s->opacity || !s->rgb || !mu_out ||
      !quat_out || !scale_out || !opacity_out || !rgb_out)
    return GS2D_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(s->quat) | reinterpret_cast<uintptr_t>(quat_out)) & 15)
    return GS2D_ERR_INVALID_ARG;
  gs2d_map_state si = st ? *st : gs2d_map_state{nullptr, nullptr, nullptr, nullptr};
  gs2d_map_state so = st_out ? *st_out : gs2d_map_state{nullptr, nullptr, nullptr, nullptr};
  // a state array is copied only when both sides give it
  if (!so.delta) si.delta = nullptr;
  if (!so.t_c) si.t_c = nullptr;
  if (!so.d_c) si.d_c = nullptr;
  if (!so.t_l) si.t_l = nullptr;
  const int nb = (n + kCompactBlock - 1) / kCompactBlock;
  int32_t* blk = static_cast<int32_t*>(workspace);
  compact_count_kernel<<<nb, kMapThreads, 0, cs>>>(keep, n, blk);
  GS2D_LAUNCH_CHECK();
  const bool scan = nb > kSelfSumBlocks;
  if (scan) {
    compact_scan_kernel<<<1, kMapThreads, 0, cs>>>(blk, nb, n_out);
    GS2D_LAUNCH_CHECK();
  }
  compact_scatter_kernel<<<nb, kMapThreads, 0, cs>>>(keep, n, blk, nb, n_out, scan ? 1 : 0, *s, si,
                                                     mu_out, quat_out, scale_out, opacity_out,
                                                     rgb_out, so, new_index);
  GS2D_LAUNCH_CHECK();
  return GS2D_OK;
}

}  // extern "C"
