// common.cuh -- constants and small device helpers shared by the kernels.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <utility>

#include "../../include/simsd.h"

namespace simsd {

constexpr uint8_t kSectData = SIMSD_SECT_DATA;
constexpr uint8_t kSectMask = SIMSD_SECT_MASK;
constexpr uint8_t kSectPad = SIMSD_SECT_PAD;

__device__ __forceinline__ void raise_error(int32_t* err_word, uint32_t bit) {
  if (err_word) atomicOr(reinterpret_cast<int*>(err_word), static_cast<int>(bit));
}

// Eq. (1) in one comparison.  Row slot i (section si, label ti) sees new
// column slot j (sj, tj) iff both are real slots and
//   (j is a data slot) == (tj < ti + [i is a data slot]).
// Data row: data columns with tj <= ti, mask columns with tj > ti.
// Mask row: data columns with tj < ti, mask columns with tj >= ti.
__host__ __device__ __forceinline__ bool temporal_visible(uint8_t si, int ti, uint8_t sj, int tj) {
  if (si == kSectPad || sj == kSectPad) return false;
  const int bias = (si == kSectData) ? 1 : 0;
  return (sj == kSectData) == (tj < ti + bias);
}

// The visibility word of a row of slot `s` (bit t: new slot t < S <= 64), for
// the 32 rows of a warp at once.  The slots of a warp's rows are consecutive:
// for each of them lane j judges columns j and j + 32, and two ballots make
// the word.  All lanes call it; rows past the last slot get 0.  (A row at a
// time, each thread walking the S labels, cost 3.4 us at S = 64.)
__device__ __forceinline__ unsigned long long slot_visibility(const int32_t* tau, const uint8_t* sect, int S, int s) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, j0 = lane, j1 = lane + 32;
  const uint8_t c0 = j0 < S ? sect[j0] : kSectPad, c1 = j1 < S ? sect[j1] : kSectPad;
  const int t0 = j0 < S ? tau[j0] : 0, t1 = j1 < S ? tau[j1] : 0;
  const int lo = __shfl_sync(full, s, 0), hi = min(S - 1, __shfl_sync(full, s, 31));
  unsigned long long vis = 0ull;
#pragma unroll 2
  for (int k = lo; k <= hi; ++k) {
    const uint8_t sk = sect[k];
    const int tk = tau[k];
    const unsigned w0 = __ballot_sync(full, temporal_visible(sk, tk, c0, t0));
    const unsigned w1 = __ballot_sync(full, temporal_visible(sk, tk, c1, t1));
    if (k == s) vis = static_cast<unsigned long long>(w1) << 32 | w0;
  }
  return vis;
}

// ---- programmatic dependent launch.  Every kernel of the library is
// launched so that it may start (set-up only) while the previous kernel on
// the stream finishes: it calls pdl_wait() before it reads or writes any
// memory that earlier work may touch, and pdl_launch_next() to let the next
// kernel be scheduled (one thread per CTA is enough).  The wait returns once
// the previous grid has completed and its memory operations are visible.
// Short kernels trigger at once; the attention and acceptance kernels only
// after their main loop, since CTAs of the next kernel that wait beside a
// long-running one slowed it down.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Host side: launches kern with the attribute that allows the overlap above
// (and a cluster dimension when cluster > 1).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_overlapped(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                     unsigned cluster, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  unsigned na = 0;
  attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[na].val.programmaticStreamSerializationAllowed = 1;
  ++na;
  if (cluster > 1) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = cluster;
    attr[na].val.clusterDim.y = 1;
    attr[na].val.clusterDim.z = 1;
    ++na;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

// ---- rotary position embedding (Su et al., RoFormer), rotate-half layout:
// for i < d/2 the pair (x_i, x_{i+d/2}) turns by the angle pos * theta^(-2i/d).
// The per-pair frequencies theta^(-2i/d) / pi come in a RopeTable (kernels.h).

// sin and cos of pi * pos * f for 0 <= pos < 2^24.  Angles are counted in
// half turns: the product is kept in float-float (the rounding error of p * hi
// comes back exactly from an FMA) and whole turns are subtracted exactly (an
// even integer from a float of at least its last place), so only r + b and
// the sine and cosine themselves round.  sincospi needs no further range
// reduction: sincosf spends most of its instructions on one, with a branch to
// local memory for huge arguments that never come here.
__device__ __forceinline__ void rope_sincos(int pos, float2 f, float* sn, float* cs) {
  const float p = static_cast<float>(pos);
  const float a = p * f.x;
  const float b = fmaf(p, f.y, fmaf(p, f.x, -a));
  const float r = fmaf(-2.0f, rintf(0.5f * a), a);
  sincospif(r + b, sn, cs);
}

// Rotates one pair in place.
__device__ __forceinline__ void rope_pair(float& x, float& y, float sn, float cs) {
  const float x2 = x * cs - y * sn;
  const float y2 = fmaf(x, sn, y * cs);
  x = x2;
  y = y2;
}

}  // namespace simsd
