// rope_tile.cuh -- the RoPE prologue of the bf16 attention kernels (Sec. 3.1
// "Position Encoding Alignment"): the query rows and the new keys of a unit
// are rotated in shared memory, in the 128-byte-swizzled halves that TMA
// wrote, before the first S = Q K^T reads them.
//
// The work is laid out by angle, not by row: a thread takes four frequencies
// of one slot (16 threads a slot), forms their sines and cosines once and
// turns that slot's g query rows and its new key with them.  One query row a
// thread, each forming all 64 pairs' angles, was bound by the sine and cosine
// instructions.  Measured, a call without -> with rotation, in the kernels
// that had the row layout and in today's (which are faster without it, too),
// 32/8 heads: 8 sequences of 512 to 2048 keys, 8 drafts (64 rows) 20.1 -> 38.8
// and 14.8 -> 17.9 us, 16 drafts (128 rows) 22.6 -> 42.3 and 19.3 -> 22.3; 19
// of 190 to 3000 keys, 7 drafts 41.7 -> 80.2 and 32.0 -> 34.1; 32 x 4096 keys,
// 16 drafts 95.3 -> 139.5 and 87.5 -> 91.9; 32 drafts, 32 sequences of 2048 to
// 8192 keys (256 rows, once per piece of a unit) 188 -> 240 and 173 -> 194.
#pragma once
#include "common.cuh"
#include "kernels.h"
#include "ptx.cuh"

namespace simsd {

constexpr int kRopeThreadsPerSlot = 16;  // 4 of the 64 pairs each

// Rotates pairs 4 q4 .. 4 q4 + 3 of row r: x_i in half h0, x_{i+64} in h1
// (row r's 16-byte chunk c sits at chunk c ^ (r & 7)).
__device__ __forceinline__ void rope_rotate4(uint8_t* h0, uint8_t* h1, int r, int q4, const float (&sn)[4],
                                             const float (&cs)[4]) {
  const int off = r * 128 + (((q4 >> 1) ^ (r & 7)) << 4) + ((q4 & 1) << 3);
  uint2* pa = reinterpret_cast<uint2*>(h0 + off);
  uint2* pb = reinterpret_cast<uint2*>(h1 + off);
  uint2 va = *pa, vb = *pb;
  float x0 = __uint_as_float(va.x << 16), x1 = __uint_as_float(va.x & 0xffff0000u);
  float x2 = __uint_as_float(va.y << 16), x3 = __uint_as_float(va.y & 0xffff0000u);
  float y0 = __uint_as_float(vb.x << 16), y1 = __uint_as_float(vb.x & 0xffff0000u);
  float y2 = __uint_as_float(vb.y << 16), y3 = __uint_as_float(vb.y & 0xffff0000u);
  rope_pair(x0, y0, sn[0], cs[0]);
  rope_pair(x1, y1, sn[1], cs[1]);
  rope_pair(x2, y2, sn[2], cs[2]);
  rope_pair(x3, y3, sn[3], cs[3]);
  va = make_uint2(pack_bf16x2(x0, x1), pack_bf16x2(x2, x3));
  vb = make_uint2(pack_bf16x2(y0, y1), pack_bf16x2(y2, y3));
  *pa = va;
  *pb = vb;
}

// Sines and cosines of pairs 4 q4 .. 4 q4 + 3 at position pos.
__device__ __forceinline__ void rope_angles4(int pos, const float2 (&f)[4], float (&sn)[4], float (&cs)[4]) {
#pragma unroll
  for (int e = 0; e < 4; ++e) rope_sincos(pos, f[e], &sn[e], &cs[e]);
}

}  // namespace simsd
