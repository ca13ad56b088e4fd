// attention_tc.cuh -- what the two one-row-block bf16 attention kernels share
// (attention_tc.cu: up to 128 query rows; attention_tc64.cu: up to 64): the
// launch parameters, the sizes and the merge of a unit's prefix splits in
// their cluster.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "common.cuh"
#include "kernels.h"
#include "ptx.cuh"

namespace simsd {

constexpr int kTile = 64;                  // keys per tile
constexpr int kD = 128;                    // head dimension
constexpr int kRows = 128;                 // MMA M
constexpr int kHalfBytes = kTile * 128;    // 64 rows x 64 bf16 (one d-half of K or V)
constexpr int kPageCache = 512;            // page ids of one sequence kept in shared memory
constexpr float kRescaleThreshold = 8.0f;  // log2 units: rescale when the max grows by > 2^8
// Split merge in place (fused): per-row partials in shared memory, padded rows
constexpr int kMaxSplitFuse = 8;              // cluster of at most 8 splits
constexpr int kPartStride = kD + 4;           // floats per partial row (no bank conflicts)
constexpr int kPartMl = kRows * kPartStride;  // (m, l) per row
constexpr int kPartWts = kPartMl + 2 * kRows;  // merge weights and output row of each row a CTA merges
constexpr int kWtsStride = kMaxSplitFuse + 1;

struct TcParams {
  const int32_t* block_table;
  const int32_t* prefix_len;
  const int32_t* tau;
  const uint8_t* section;
  const int32_t* rope_pos;  // [Bt][2*gamma] or null (inputs rotated already)
  __nv_bfloat16* out;
  float* ws;  // partials: O [units*nsplit][rows_blk][128] then (m, l) [units*nsplit][rows_blk][2]
  int32_t* err_word;
  int max_pages, page_size, num_pages;
  int Bt, gamma, S, Hq, Hkv, g, rb, rows_blk, s_blk, nsplit;
  int sort;  // order sequences longest prefix first (grids of more than one wave)
  int slots;  // CTAs resident at once: blocks past this start in a later wave
  int fuse;   // the prefix splits of a unit form a cluster and merge in shared memory
  float scale_log2;
  // bounded waits: time limit and extra arrivals expected on bar_p (0 in
  // normal use; a test arms one launch so that a wait runs out)
  unsigned long long wait_ns;
  uint32_t extra_p;
  RopeTable rope;
};

// Merge of the splits of a unit in their cluster (128 threads, warps 0-3):
// O = sum_i 2^(m_i - M) O_i / sum_i 2^(m_i - M) l_i.  CTA `split` takes rows
// split, split + nsplit, ... of the row block.  The partial O of a warp's
// first U rows (a row per warp, lanes over d) are requested from every split
// first; while they travel, thread k forms row k's weights from its (m, l)
// pairs.  With every lane forming its row's weights itself the merge was
// bound by those instructions (one warp a scheduler): 2.1 to 3.4 us.  Every
// thread arrives on the cluster barrier once its remote loads have returned;
// the caller waits on it.
template <int NS, int U>
__device__ __forceinline__ void merge_splits(const TcParams& p, float* part, int split, int rblk, int b, int kvh) {
  const int nsp = p.nsplit, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nrows = (p.rows_blk - split + nsp - 1) / nsp;
  uint32_t peer[NS];
#pragma unroll
  for (int i = 0; i < NS; ++i) peer[i] = peer_smem(smem_u32(part), min(i, nsp - 1));
  float4 x[U][NS];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int i = 0; i < NS; ++i)
        if (i < nsp && k0 + 4 * u < nrows)
          x[u][i] = ld_cluster_f32x4(peer[i] + 4 * ((split + (k0 + 4 * u) * nsp) * kPartStride + 4 * lane));
  };
  fetch(warp);
  float* wts = part + kPartWts;  // [row of this CTA][NS weights, output offset]
  if (tid < nrows) {
    const int r = split + tid * nsp;
    float m[NS], l[NS], M = -INFINITY, L = 0.f;
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      m[i] = -INFINITY;
      l[i] = 0.f;
      if (i < nsp) ld_cluster_f32x2(peer[i] + 4 * (kPartMl + 2 * r), m[i], l[i]);
    }
    const int sl = r / p.g, sr = rblk * p.s_blk + sl;
#pragma unroll
    for (int i = 0; i < NS; ++i)
      if (l[i] > 0.f) M = fmaxf(M, m[i]);
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      m[i] = (M != -INFINITY && l[i] > 0.f) ? exp2f(m[i] - M) : 0.f;
      L = fmaf(m[i], l[i], L);
    }
    const float inv = L > 0.f ? 1.f / L : 0.f;
#pragma unroll
    for (int i = 0; i < NS; ++i) wts[tid * kWtsStride + i] = m[i] * inv;
    // the row's place in the output, in rows of d (-1: past the last slot)
    wts[tid * kWtsStride + kMaxSplitFuse] =
        __int_as_float(sr < p.S ? (b * p.S + sr) * p.Hq + kvh * p.g + (r - sl * p.g) : -1);
  }
  asm volatile("bar.sync 2, 128;" ::: "memory");
#pragma unroll 1
  for (int k0 = warp; k0 < nrows; k0 += 4 * U) {
    if (k0 != warp) fetch(k0);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = k0 + 4 * u;
      if (k >= nrows) break;
      const float* w = wts + k * kWtsStride;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int i = 0; i < NS; ++i) {
        if (i < nsp) {
          const float wi = w[i];
          v.x = fmaf(wi, x[u][i].x, v.x);
          v.y = fmaf(wi, x[u][i].y, v.y);
          v.z = fmaf(wi, x[u][i].z, v.z);
          v.w = fmaf(wi, x[u][i].w, v.w);
        }
      }
      const int at = __float_as_int(w[kMaxSplitFuse]);
      if (at >= 0)
        reinterpret_cast<uint2*>(p.out + static_cast<size_t>(at) * kD)[lane] =
            make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
    }
  }
  cluster_arrive();
}

// The caller's dispatch over the number of splits: at most 16 float4 of a
// lane in flight (all the rows of a warp at 64 rows and 2 or 4 splits).
__device__ __forceinline__ void merge_unit(const TcParams& p, float* part, int split, int rblk, int b, int kvh) {
  if (p.nsplit <= 2)
    merge_splits<2, 8>(p, part, split, rblk, b, kvh);
  else if (p.nsplit <= 4)
    merge_splits<4, 4>(p, part, split, rblk, b, kvh);
  else
    merge_splits<8, 2>(p, part, split, rblk, b, kvh);
}

// The kernel of row blocks of at most 64 query rows (attention_tc64.cu).
constexpr int kTc64Rows = 64;
cudaError_t launch_attention_tc64(const CUtensorMap& tq, const CUtensorMap& tkn, const CUtensorMap& tvn,
                                  const CUtensorMap& tkc, const CUtensorMap& tvc, const TcParams& p,
                                  cudaStream_t stream);

}  // namespace simsd
