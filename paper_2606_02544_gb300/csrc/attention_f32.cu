// attention_f32.cu -- fp32 verification attention on CUDA cores (the paper's
// own runs are fp32, Sec. 4.1).
//
// Work unit: (sequence b, KV head, row block, key range).  The g * 2*gamma
// query rows that share a KV head are packed 8 to a warp, up to eight warps a
// row block, so every K/V row is read once for all of them (one CTA per query
// row re-read the whole cache 16 to 256 times through L2: 8 sequences of 512
// to 1024 keys, 16/8 heads, 4 drafts, d 128 took 149 us against 23.0 us here;
// 8 of 1024 to 2048 keys, 32/8 heads, 16 drafts 1789 against 255; one of 4096
// keys, 16/8 heads, 4 drafts 155 against 38.1).  What bounds it, by counters:
// the first (2.2 TB/s, 13 warps an SM) issues in 33% of the cycles, its warps
// waiting for one another at the cluster barriers (ranges of unequal length),
// for fixed latencies and for K and V; the second (25 TFLOP/s, nine warps on
// each of 128 SMs) issues in 43% with the FMA pipe 54% busy and waits for
// shared-memory loads.  Keys come in tiles of 32: the paged prefix rows, then
// the new slots admitted by Eq. (1).  A producer warp fetches them, lane i key
// i's row with one bulk copy, into rows padded against bank conflicts.
//   S = Q K^T  a lane owns two keys (k, k + 16) and four of the warp's rows
//              (the half-warps take the even and the odd ones): per 4
//              elements of d two 16-byte loads of K and four broadcast loads
//              of Q feed 16 packed FMAs (even and odd elements summed apart).
//   O += P V   a lane owns d/32 columns of the 8 rows: per key one load of V
//              and two broadcast loads of P (written by the lanes as
//              [key][row]) feed the packed FMAs, rows in pairs (columns in
//              pairs would need every P twice: 15% slower at 32 x 1500 keys).
// The running maximum lags: it is raised only when some score exceeds it by
// more than 8 (a warp vote), so row maxima and the rescale of O are rare; the
// sums stay one per lane until the end.  K of the next tile loads while this
// one's P V runs, V while its S does; the warps of a row block pass one
// another freely, and several CTAs share an SM.
//
// Few units: the key tiles of a unit are dealt over the CTAs of a cluster (up
// to 16), which merge their partial (O, m, l) through distributed shared
// memory.  When the inputs are not rotated yet (Sec. 3.1 RoPE copy), query
// rows and new keys are rotated in shared memory; cached keys are stored
// rotated.
//
// Every mbarrier wait is bounded (a consumer's also ends with the producer's,
// through the abort flag): one that expires sets SIMSD_EW_TIMEOUT, the CTA
// leaves its loops, waits for its own copies and finishes (its output is
// undefined).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <map>
#include <mutex>

#include "common.cuh"
#include "kernels.h"
#include "ptx.cuh"

namespace cg = cooperative_groups;

namespace simsd {
namespace {
constexpr int kF32Rows = 8;      // query rows of a warp
constexpr int kF32Keys = 32;     // keys of a tile
constexpr int kF32MaxWarps = 8;  // row groups of a row block (then the producer warp)
constexpr int kF32MaxSplit = 16;  // key ranges of a unit (cluster size)
constexpr int kF32Merge = 4;     // ranges merged at a time
constexpr int kF32GridY = 65535;  // most blocks of a grid in y
constexpr int kF32Regs = 112;    // 18 warps an SM by the register file
// shared memory: of an SM, of one CTA (dynamic), and of a CTA beside its
// dynamic part (static and reserved, rounded up)
constexpr size_t kF32SmSmem = 233472, kF32MaxSmem = 226 * 1024, kF32Static = 2200;
constexpr float kF32Lag = 8.0f;  // natural-log units the running maximum may lag behind

// Dynamic shared memory (floats) of a CTA with W row groups.  Rows are padded
// by 16 bytes: 8 lanes reading one 16-byte column of 8 rows, and the even and
// odd rows the half-warps read, then fall into different banks.
template <int D>
struct F32Layout {
  static constexpr int kRow = D + 4;
  static constexpr int kV = kF32Keys * kRow;      // [32][kRow], after K's
  static constexpr int kQ = 2 * kF32Keys * kRow;  // [8 W][kRow]
  __host__ __device__ static constexpr int p(int W) { return kQ + kF32Rows * W * kRow; }  // [W][32][8]; then (m, l)
  __host__ __device__ static constexpr size_t bytes(int W) {
    return static_cast<size_t>(p(W) + W * kF32Keys * kF32Rows) * sizeof(float);
  }
};

// Row of the warp at position i of a lane's four (half-warp h), and of
// position x of a key's eight P values [half][4].
__device__ __forceinline__ constexpr int row_of(int h, int i) { return 2 * i + h; }
__device__ __forceinline__ constexpr int row_at(int x) { return 2 * (x & 3) + (x >> 2); }

template <int D>
__global__ void __maxnreg__(kF32Regs)
    attention_f32_kernel(const __grid_constant__ AttnF32Args a, int rb, int nsplit) {
  using L = F32Layout<D>;
  constexpr int NC = D / 32;  // columns of a lane in O
  constexpr int KR = L::kRow;
  constexpr uint32_t kRowBytes = D * sizeof(float);
  constexpr int kChunks = D / 4;          // 16-byte pieces of a row
  constexpr int kPerCopy = 32 / kChunks;  // rows a warp's copy covers, a piece a lane
  extern __shared__ __align__(16) float smem[];
  __shared__ __align__(8) uint64_t bar_k, bar_v, bar_kfree, bar_vfree;
  __shared__ int lab_tau[64], lab_pos[64];
  __shared__ uint8_t lab_sect[64];
  __shared__ int bad_sh, abort_sh;
  __shared__ int asked[2];  // tiles of K and of V requested
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int W = (blockDim.x >> 5) - 1;  // consumer warps
  const bool producer = warp == W;
  const int half = lane >> 4, kp = lane & 15;
  const unsigned full = 0xffffffffu;
  volatile int* abort_flag = &abort_sh;
  // KV heads lie over y and z, each of which ends at 65535 (in x the divisions
  // that find one cost 0.2 us a call); the last z may not be full
  const int kvh = blockIdx.z * kF32GridY + blockIdx.y;
  if (kvh >= a.Hkv) return;  // (a whole cluster)
  if (tid == 0) {
    bad_sh = 0;
    abort_sh = 0;
    mbar_init(smem_u32(&bar_k), 1);
    mbar_init(smem_u32(&bar_v), 1);
    mbar_init(smem_u32(&bar_kfree), a.k_release);
    mbar_init(smem_u32(&bar_vfree), W);
    fence_mbar_init();
  }
  __syncthreads();
  pdl_wait();
  const int S = 2 * a.gamma, g = a.Hq / a.Hkv, R = S * g;
  // grid: (sequence, row block, split) x KV head; the splits of a unit are
  // adjacent (a cluster), then its row blocks (which share its K/V in L2)
  const unsigned bx = blockIdx.x / static_cast<unsigned>(nsplit);
  const int split = blockIdx.x - bx * nsplit;
  const int b = bx / static_cast<unsigned>(rb), rblk = bx - b * rb;
  const int blk_row0 = rblk * W * kF32Rows;    // the CTA's first row of the unit
  const int row0 = blk_row0 + warp * kF32Rows;  // this warp's

  const int n = a.prefix_len[b];
  const int32_t* bt = a.block_table + static_cast<size_t>(b) * a.max_pages;
  const bool n_bad = n < 0 || static_cast<long long>(n) > static_cast<long long>(a.max_pages) * a.page_size;
  const int nkeys = n_bad ? 0 : n + S;
  const int T = (nkeys + kF32Keys - 1) / kF32Keys;
  auto q_offset = [&](int r) {  // row r of the unit in q and out
    const int s = r / g;
    return ((static_cast<size_t>(b) * S + s) * a.Hq + kvh * g + (r - s * g)) * D;
  };
  if (producer) {
    // range `split` takes tiles split, split + nsplit, ...: its first tile
    // does not depend on the prefix length, so the page ids of that tile are
    // loaded beside it (and not used past it)
    const int pi0 = (split * kF32Keys + lane) / a.page_size;
    const int page0 = pi0 < a.max_pages ? bt[pi0] : -1;
    // keys 0..n-1 are the prefix rows, keys n..n+S-1 the new slots; lane i finds
    // key i of a tile.  Slots of padding are no row's key: their rows are zeros,
    // as are rows past the last key and pages out of range.  src: 1 cache, 2 new
    // slots, 0 none.
    auto locate = [&](int t, long long& off) -> int {
      const int j = t * kF32Keys + lane;
      if (j < n) {
        const int pi = j / a.page_size;
        const int pg = t == split ? page0 : bt[pi];
        if (pg < 0 || pg >= a.num_pages) return 0;
        off = ((static_cast<long long>(pg) * a.Hkv + kvh) * a.page_size + (j - pi * a.page_size)) * D;
        return 1;
      }
      if (j < nkeys && a.section[static_cast<size_t>(b) * S + (j - n)] != kSectPad) {
        off = ((static_cast<long long>(b) * S + (j - n)) * a.Hkv + kvh) * D;
        return 2;
      }
      return 0;
    };
    // one bulk copy per key; the rows of missing keys become zeros before the
    // arrival that lets the tile complete
    auto load_tile = [&](float* dst, const float* cache, const float* fresh, uint64_t* bar, long long off, int src) {
      const unsigned have = __ballot_sync(full, src != 0);
      if (src == 0)
        for (int c = 0; c < D / 4; ++c)
          *reinterpret_cast<float4*>(dst + lane * KR + 4 * c) = make_float4(0.f, 0.f, 0.f, 0.f);
      __syncwarp();
      if (lane == 0) mbar_arrive_expect_tx(smem_u32(bar), static_cast<uint32_t>(__popc(have)) * kRowBytes);
      __syncwarp();
      if (src != 0) bulk_load(smem_u32(dst + lane * KR), (src == 2 ? fresh : cache) + off, kRowBytes, smem_u32(bar));
    };
    bool ok = true;
    int it = 0, nk = 0, nv = 0;
    for (int t = split; ok && t < T; t += nsplit, ++it) {
      long long off = 0;
      const int src = locate(t, off);
      ok = it == 0 || mbar_wait_warp(smem_u32(&bar_kfree), (it - 1) & 1, abort_flag, a.wait_ns);
      if (ok) {
        load_tile(smem, a.k_cache, a.k_new, &bar_k, off, src);
        ++nk;
      }
      ok = ok && (it == 0 || mbar_wait_warp(smem_u32(&bar_vfree), (it - 1) & 1, abort_flag, a.wait_ns));
      if (ok) {
        load_tile(smem + L::kV, a.v_cache, a.v_new, &bar_v, off, src);
        ++nv;
      }
    }
    if (lane == 0) {
      asked[0] = nk;
      asked[1] = nv;
      if (!ok) *abort_flag = 1;
    }
  } else {
    // this warp's query rows (zeros past the unit's last), waited for below.
    // The producer's bulk copies, one a row and 58 cycles each to issue, held
    // up the first K: 128 rows of d 64 over 24 keys 9.9 -> 8.3 us a call, 8
    // sequences of 64 rows a KV head over 128 keys 21.3 -> 19.6.
    {
      float* qs = smem + L::kQ + warp * kF32Rows * KR;
      const int own = min(row0 + (lane & (kF32Rows - 1)), R - 1);
      const unsigned long long from = reinterpret_cast<unsigned long long>(a.q + q_offset(own));
      const int sub = lane / kChunks, col = 4 * (lane % kChunks);
#pragma unroll
      for (int i = 0; i < kF32Rows; i += kPerCopy) {
        const int r = i + sub;
        const float* row = reinterpret_cast<const float*>(__shfl_sync(full, from, r));
        cp_async16(smem_u32(qs + r * KR + col), row + col, row0 + r < R ? 16u : 0u);
      }
    }
    // slot labels, and every page the sequence needs is checked, while the
    // first loads are in flight
    const int nt = 32 * W;
    for (int t = tid; t < S; t += nt) {
      lab_tau[t] = a.tau[static_cast<size_t>(b) * S + t];
      lab_sect[t] = a.section[static_cast<size_t>(b) * S + t];
      lab_pos[t] = a.rope_pos ? a.rope_pos[static_cast<size_t>(b) * S + t] : 0;
    }
    if (n_bad) {
      if (tid == 0 && split == 0 && rblk == 0 && kvh == 0) raise_error(a.err_word, SIMSD_EW_PREFIX_LEN);
    } else {
      const int npages = (n + a.page_size - 1) / a.page_size;
      bool bad = false;
      for (int p = tid; p < npages; p += nt) {
        const int pg = bt[p];
        bad |= pg < 0 || pg >= a.num_pages;
      }
      if (bad) {
        bad_sh = 1;
        if (split == 0 && rblk == 0 && kvh == 0) raise_error(a.err_word, SIMSD_EW_PAGE);
      }
    }
    asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory");
  }

  // m, l: rows row_of(half, i) of the warp; o: P positions 2q and 2q + 1
  float m[4], l[4];
  unsigned long long o[4][NC];
  unsigned act_rows = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    m[i] = -INFINITY;
    l[i] = 0.f;
#pragma unroll
    for (int c = 0; c < NC; ++c) o[i][c] = 0ull;
  }
  if (!producer) {
  const bool seq_bad = n_bad || bad_sh != 0;
  float* ks = smem;
  const float* vs = smem + L::kV;
  float* qs = smem + L::kQ + warp * kF32Rows * KR;          // this warp's rows
  float* ps = smem + L::p(W) + warp * kF32Keys * kF32Rows;  // this warp's P
  // rows of this warp that have an output to compute, and what they see of
  // the new slots (lane i < 8: row i)
  const int own_row = row0 + min(lane, kF32Rows - 1), own_slot = own_row / g;
  unsigned long long vis = slot_visibility(lab_tau, lab_sect, S, own_slot);
  const bool act = lane < kF32Rows && own_row < R && !seq_bad && lab_sect[min(own_slot, S - 1)] != kSectPad;
  if (!act) vis = 0ull;
  act_rows = __ballot_sync(full, act);
  bool ok = true;
  cp_async_wait_all();
  __syncwarp();
  if (a.rope_pos) {
    // lane i turns pairs i, i + 32, ...; rows of one slot share the angles
    float sn[D / 64], cs[D / 64];
    int prev = -1;
    for (int i = 0; i < kF32Rows && row0 + i < R; ++i) {
      const int s = (row0 + i) / g;
      if (s != prev) {
#pragma unroll
        for (int e = 0; e < D / 64; ++e) rope_sincos(lab_pos[s], a.rope.f[lane + 32 * e], &sn[e], &cs[e]);
        prev = s;
      }
#pragma unroll
      for (int e = 0; e < D / 64; ++e)
        rope_pair(qs[i * KR + lane + 32 * e], qs[i * KR + D / 2 + lane + 32 * e], sn[e], cs[e]);
    }
  }
  __syncwarp();
  uint32_t par = 0;
  for (int t = split; t < T; t += nsplit, par ^= 1) {
    const bool has_new = (t + 1) * kF32Keys > n;
    ok = ok && mbar_wait_warp(smem_u32(&bar_k), par, abort_flag);
    if (has_new && a.rope_pos) {
      // the tile's new keys are rotated in place, rows dealt over the warps
      for (int i = warp; ok && i < kF32Keys; i += W) {
        const int slot = t * kF32Keys + i - n;
        if (slot < 0 || slot >= S) continue;
#pragma unroll
        for (int e = 0; e < D / 64; ++e) {
          float sn, cs;
          rope_sincos(lab_pos[slot], a.rope.f[lane + 32 * e], &sn, &cs);
          rope_pair(ks[i * KR + lane + 32 * e], ks[i * KR + D / 2 + lane + 32 * e], sn, cs);
        }
      }
      asm volatile("bar.sync 1, %0;" ::"r"(32 * W) : "memory");
    }
    // after a wait that expired the warp runs through its tiles without
    // touching them (the other warps may meet it above)
    if (!ok) continue;
    // ---- S: keys kp and kp + 16 against rows row_of(half, 0..3)
    float x[2][4];
    {
      unsigned long long acc[2][4];
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[0][i] = acc[1][i] = 0ull;
      const float* k0 = ks + kp * KR;
      const float* q0 = qs + half * KR;
#pragma unroll 8
      for (int c = 0; c < D / 4; ++c) {
        const ulonglong2 ka = *reinterpret_cast<const ulonglong2*>(k0 + 4 * c);
        const ulonglong2 kb = *reinterpret_cast<const ulonglong2*>(k0 + 16 * KR + 4 * c);
        ulonglong2 qq[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) qq[i] = *reinterpret_cast<const ulonglong2*>(q0 + 2 * i * KR + 4 * c);
        // (the eight sums in turn: an FMA on one waits for the last on it)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          acc[0][i] = fma_f32x2(ka.x, qq[i].x, acc[0][i]);
          acc[1][i] = fma_f32x2(kb.x, qq[i].x, acc[1][i]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          acc[0][i] = fma_f32x2(ka.y, qq[i].y, acc[0][i]);
          acc[1][i] = fma_f32x2(kb.y, qq[i].y, acc[1][i]);
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          float s0, s1;
          f32x2_split(acc[e][i], s0, s1);
          x[e][i] = (s0 + s1) * a.scale;
        }
      }
    }
    // this warp is done with the tile's K
    if (has_new) fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&bar_kfree));
    // ---- visibility: every prefix key; a new slot where Eq. (1) admits it
    if (has_new) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const unsigned long long vr = __shfl_sync(full, vis, row_of(half, i));
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int slot = t * kF32Keys + kp + 16 * e - n;
          const bool see = slot < 0 || (slot < S && ((vr >> slot) & 1ull));
          x[e][i] = see ? x[e][i] : -INFINITY;
        }
      }
    }
    // ---- the running maximum, raised when some score leads it by kF32Lag
    bool lead = false;
#pragma unroll
    for (int i = 0; i < 4; ++i) lead |= fmaxf(x[0][i], x[1][i]) > m[i] + kF32Lag;
    if (__any_sync(full, lead)) {
      float f[4], fo[4];  // of this half's rows, and of the other's
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float mx = fmaxf(x[0][i], x[1][i]);
#pragma unroll
        for (int w = 8; w > 0; w >>= 1) mx = fmaxf(mx, __shfl_xor_sync(full, mx, w));
        mx = fmaxf(m[i], mx);
        f[i] = mx == -INFINITY ? 1.f : expf(m[i] - mx);
        m[i] = mx;
        l[i] *= f[i];
        fo[i] = __shfl_xor_sync(full, f[i], 16);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        // positions 2q, 2q + 1: half q >> 1, its rows 2 (q & 1) and + 1
        const bool own = (q >> 1) == half;
        const float f0 = own ? f[2 * (q & 1)] : fo[2 * (q & 1)];
        const float f1 = own ? f[2 * (q & 1) + 1] : fo[2 * (q & 1) + 1];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          float lo, hi;
          f32x2_split(o[q][c], lo, hi);
          o[q][c] = f32x2(lo * f0, hi * f1);
        }
      }
    }
    // ---- P = e^(x - m), to shared memory as [key][half][4]
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      float pv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        pv[i] = expf(x[e][i] - (m[i] == -INFINITY ? 0.f : m[i]));
        l[i] += pv[i];
      }
      // (the two chunks of a key swap every four keys: 8 lanes' stores then
      // fall into different banks)
      const int key = kp + 16 * e;
      *reinterpret_cast<float4*>(ps + key * kF32Rows + ((half ^ ((key >> 2) & 1)) << 2)) =
          make_float4(pv[0], pv[1], pv[2], pv[3]);
    }
    __syncwarp();
    ok = mbar_wait_warp(smem_u32(&bar_v), par, abort_flag);
    if (!ok) continue;
    // ---- O += P V
    auto load_v = [&](int j, float(&v)[NC]) {
      const float* p = vs + j * KR + NC * lane;
      if constexpr (NC == 4) {
        const float4 t4 = *reinterpret_cast<const float4*>(p);
        v[0] = t4.x;
        v[1] = t4.y;
        v[2] = t4.z;
        v[3] = t4.w;
      } else {
        const float2 t2 = *reinterpret_cast<const float2*>(p);
        v[0] = t2.x;
        v[1] = t2.y;
      }
    };
    auto load_p = [&](int j, unsigned long long(&pp)[4]) {
      const int sw = ((j >> 2) & 1) << 2;
      const ulonglong2 w0 = *reinterpret_cast<const ulonglong2*>(ps + j * kF32Rows + sw);
      const ulonglong2 w1 = *reinterpret_cast<const ulonglong2*>(ps + j * kF32Rows + (4 ^ sw));
      pp[0] = w0.x;
      pp[1] = w0.y;
      pp[2] = w1.x;
      pp[3] = w1.y;
    };
    // a row must not take 0 * (infinity or NaN) from a new slot it does not
    // see: a tile with such a value among its new slots takes the select below
    bool odd = false;
    if (has_new) {
      // (eight rows at a time, cached keys before the first slot among them:
      // the select is right for those too.  One row after the other to the
      // tile's end took 1900 cycles of a call of one tile a CTA; a step of one
      // sequence of 128 keys 15.7 -> 14.8 us.)
      const int j1 = min(kF32Keys, nkeys - t * kF32Keys);
#pragma unroll 1
      for (int j0 = max(0, n - t * kF32Keys) & ~7; j0 < j1; j0 += 8) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          float v[NC];
          load_v(j0 + j, v);
#pragma unroll
          for (int c = 0; c < NC; ++c) odd |= !(fabsf(v[c]) < INFINITY);
        }
      }
    }
    if (!__any_sync(full, odd)) {
#pragma unroll 8
      for (int j = 0; j < kF32Keys; ++j) {
        float v[NC];
        unsigned long long pp[4];
        load_v(j, v);
        load_p(j, pp);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const unsigned long long vv = f32x2(v[c], v[c]);
#pragma unroll
          for (int q = 0; q < 4; ++q) o[q][c] = fma_f32x2(pp[q], vv, o[q][c]);
        }
      }
    } else {
#pragma unroll 1
      for (int j = 0; j < kF32Keys; ++j) {
        float v[NC];
        unsigned long long pp[4];
        load_v(j, v);
        load_p(j, pp);
        const int slot = t * kF32Keys + j - n;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const unsigned long long v0 = __shfl_sync(full, vis, row_at(2 * q));
          const unsigned long long v1 = __shfl_sync(full, vis, row_at(2 * q + 1));
          const bool see0 = slot < 0 || (slot < S && ((v0 >> slot) & 1ull));
          const bool see1 = slot < 0 || (slot < S && ((v1 >> slot) & 1ull));
          float p0, p1;
          f32x2_split(pp[q], p0, p1);
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            float o0, o1;
            f32x2_split(o[q][c], o0, o1);
            o[q][c] = f32x2(see0 ? fmaf(p0, v[c], o0) : o0, see1 ? fmaf(p1, v[c], o1) : o1);
          }
        }
      }
    }
    // this warp is done with the tile's V
    if (has_new) fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&bar_vfree));
  }
  if (!ok && lane == 0) *abort_flag = 1;
  // ---- the lanes' sums (over the 16 lanes of a half)
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int w = 8; w > 0; w >>= 1) l[i] += __shfl_xor_sync(full, l[i], w);
    // padding rows, rows past the unit, a bad sequence
    if (!((act_rows >> row_of(half, i)) & 1u)) l[i] = 0.f;
  }
  }  // consumer warps
  pdl_launch_next();  // (the tiles are done: common.cuh)
  __syncthreads();
  if (*abort_flag) {
    // a wait expired: the copies still in flight are waited for (with the
    // full limit), so that none lands after the CTA has gone.  A tile is
    // requested after the one before has been consumed, so only the last
    // phase can be open.
    if (tid == 0) {
      raise_error(a.err_word, SIMSD_EW_TIMEOUT);
      if (asked[0] > 0) mbar_wait(smem_u32(&bar_k), (asked[0] - 1) & 1, nullptr);
      if (asked[1] > 0) mbar_wait(smem_u32(&bar_v), (asked[1] - 1) & 1, nullptr);
    }
    __syncthreads();
  }
  // (m, l) of P position x, to every lane
  auto at = [&](const float(&w)[4], int x) { return __shfl_sync(full, w[x & 3], (x >> 2) << 4); };
  auto put = [&](float* dst, const float(&y)[NC]) {
    if constexpr (NC == 4)
      *reinterpret_cast<float4*>(dst + 4 * lane) = make_float4(y[0], y[1], y[2], y[3]);
    else
      *reinterpret_cast<float2*>(dst + 2 * lane) = make_float2(y[0], y[1]);
  };
  // O of position x times f (zeros when the row has no sum)
  auto o_row = [&](int x, bool any, float f, float(&y)[NC]) {
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      float lo, hi;
      f32x2_split(o[x >> 1][c], lo, hi);
      y[c] = any ? ((x & 1) ? hi : lo) * f : 0.f;
    }
  };
  if (nsplit == 1) {
    if (producer) return;
#pragma unroll
    for (int x = 0; x < kF32Rows; ++x) {
      const int r = row0 + row_at(x);
      const float lx = at(l, x);
      if (r >= R) continue;
      float y[NC];
      o_row(x, lx != 0.f, 1.f / lx, y);
      put(a.out + q_offset(r), y);
    }
    return;
  }
  // ---- merge of the unit's key ranges: O = sum_i e^(m_i - M) O_i / sum_i
  // e^(m_i - M) l_i.  Partial O replaces K and V, (m, l) the P region (every
  // warp of the CTA is done with them).
  cg::cluster_group cluster = cg::this_cluster();
  const int rows_cta = kF32Rows * W;
  static_assert(kF32MaxWarps * kF32Rows <= 2 * kF32Keys, "the partial O fits the K and V tiles");
  float* part_ml = smem + L::p(W);  // [8 W][2]
  if (!producer) {
    float* part = smem + warp * kF32Rows * KR;
#pragma unroll
    for (int x = 0; x < kF32Rows; ++x) {
      const float lx = at(l, x), mx = at(m, x);
      const bool any = lx != 0.f;
      float y[NC];
      o_row(x, any, 1.f, y);
      put(part + row_at(x) * KR, y);
      if (lane == 0)
        *reinterpret_cast<float2*>(part_ml + 2 * (warp * kF32Rows + row_at(x))) =
            make_float2(any ? mx : -INFINITY, any ? lx : 0.f);
    }
  }
  cluster.sync();
  // CTA c takes rows c, c + nsplit, ... of the block; a thread takes 16-byte
  // columns.  The ranges go kF32Merge at a time, loaded together and folded
  // into a running (M, L, O).
  const int mine = (rows_cta - split + nsplit - 1) / nsplit;
  for (int task = tid; task < mine * (D / 4); task += blockDim.x) {
    const int r = split + (task / (D / 4)) * nsplit, c4 = task % (D / 4);
    if (blk_row0 + r >= R) continue;
    const uint32_t ml_at = smem_u32(part_ml + 2 * r), o_at = smem_u32(smem + r * KR + 4 * c4);
    float M = -INFINITY, Ls = 0.f;
    float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (int i0 = 0; i0 < nsplit; i0 += kF32Merge) {
      float mi[kF32Merge], li[kF32Merge];
      float4 ov[kF32Merge];
#pragma unroll
      for (int i = 0; i < kF32Merge; ++i) {
        const int from = min(i0 + i, nsplit - 1);  // (past the end: read again, not used)
        ld_cluster_f32x2(peer_smem(ml_at, from), mi[i], li[i]);
        ov[i] = ld_cluster_f32x4(peer_smem(o_at, from));
        if (i0 + i >= nsplit) li[i] = 0.f;
      }
      float Mn = M;
#pragma unroll
      for (int i = 0; i < kF32Merge; ++i) Mn = fmaxf(Mn, li[i] != 0.f ? mi[i] : -INFINITY);
      const float f = Ls != 0.f ? expf(M - Mn) : 0.f;
      Ls *= f;
      y = make_float4(y.x * f, y.y * f, y.z * f, y.w * f);
      M = Mn;
#pragma unroll
      for (int i = 0; i < kF32Merge; ++i) {
        const float w = li[i] != 0.f ? expf(mi[i] - M) : 0.f;
        Ls = fmaf(w, li[i], Ls);
        y.x = fmaf(w, ov[i].x, y.x);
        y.y = fmaf(w, ov[i].y, y.y);
        y.z = fmaf(w, ov[i].z, y.z);
        y.w = fmaf(w, ov[i].w, y.w);
      }
    }
    const float inv = Ls != 0.f ? 1.f / Ls : 0.f;
    *reinterpret_cast<float4*>(a.out + q_offset(blk_row0 + r) + 4 * c4) =
        make_float4(y.x * inv, y.y * inv, y.z * inv, y.w * inv);
  }
  cluster.sync();  // no CTA leaves while a peer may still read its partials
}

// Dynamic shared memory at which at most k CTAs of W row groups fit an SM.
// Asking for more than the kernel uses spreads a grid: CTAs of a cluster (and
// clusters of a grid) otherwise pack the first SMs and GPCs as full as they
// fit (64 units in 8 ranges on 152 SMs, room for 5 CTAs an SM: 30.2 us; room
// for the 4 that an even spread needs: 25.3).
template <int D>
size_t smem_for(int W, int k) {
  return std::max(F32Layout<D>::bytes(W), std::min(kF32MaxSmem, (kF32SmSmem / k - kF32Static) & ~size_t{15}));
}

// How many clusters of ns CTAs (W row groups, at most k CTAs an SM) are
// resident at once, asked once per device, shape and size from the occupancy
// calculator: a cluster lies within a GPC, so fewer fit than SMs x k / ns.
template <int D>
cudaError_t resident_clusters(int W, int k, int ns, int* out) {
  static std::mutex mu;
  static bool attr[64] = {};
  static std::map<std::array<int, 4>, int> known;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(mu);
  if (!attr[dev]) {
    e = cudaFuncSetAttribute(attention_f32_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(kF32MaxSmem));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(attention_f32_kernel<D>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    attr[dev] = true;
  }
  const std::array<int, 4> key{dev, W, k, ns};
  const auto it = known.find(key);
  if (it != known.end()) {
    *out = it->second;
    return cudaSuccess;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(ns));
  cfg.blockDim = dim3(32 * (W + 1));
  cfg.dynamicSmemBytes = smem_for<D>(W, k);
  cudaLaunchAttribute la[1];
  la[0].id = cudaLaunchAttributeClusterDimension;
  la[0].val.clusterDim.x = static_cast<unsigned>(ns);
  la[0].val.clusterDim.y = 1;
  la[0].val.clusterDim.z = 1;
  cfg.attrs = la;
  cfg.numAttrs = 1;
  e = cudaOccupancyMaxActiveClusters(out, attention_f32_kernel<D>, &cfg);
  if (e == cudaSuccess) known[key] = *out;
  return e;
}

template <int D>
cudaError_t launch(AttnF32Args a, cudaStream_t stream, const WaitFault& fault) {
  // row groups of 8, at most eight to a row block, spread evenly over the blocks
  const int groups = (2 * a.gamma * (a.Hq / a.Hkv) + kF32Rows - 1) / kF32Rows;
  const int rb = (groups + kF32MaxWarps - 1) / kF32MaxWarps;
  const int W = (groups + rb - 1) / rb;
  const long long units = static_cast<long long>(a.Bt) * a.Hkv * rb;
  const long long tiles = (static_cast<long long>(a.max_pages) * a.page_size + 2 * a.gamma + kF32Keys - 1) / kF32Keys;
  // Key ranges: the most that keep the whole grid resident at once with about
  // ten consumer warps an SM (a second CTA of eight halves the first's rate:
  // 32 units of 64 rows took 38.6 us in 4 ranges, one CTA an SM, and 60.8 in
  // 8; 16 units 27.9 us in 6 ranges and 38.8 in 8, of which one GPC holds
  // only two) and at least one tile each.
  int full = 0;  // (also sets the kernel's attributes)
  cudaError_t e = resident_clusters<D>(W, 1, 1, &full);
  if (e != cudaSuccess) return e;
  const int room = std::max(1, std::min<int>(10 / W, static_cast<int>(kF32SmSmem / (F32Layout<D>::bytes(W) + kF32Static))));
  int ns = static_cast<int>(std::min<long long>({kF32MaxSplit, tiles, a.num_sms * room / units}));
  int k = room;
  for (; ns > 1; --ns) {
    int fit = 0;
    // the CTAs an SM an even spread needs, or one more where GPCs hold fewer
    k = std::min<int>(room, static_cast<int>((units * ns + a.num_sms - 1) / a.num_sms));
    for (; k <= room; ++k) {
      e = resident_clusters<D>(W, k, ns, &fit);
      if (e != cudaSuccess) return e;
      if (fit >= units) break;
    }
    if (fit >= units) break;
  }
  ns = std::max(ns, 1);
  a.wait_ns = fault.wait_ns ? fault.wait_ns : kWaitLimitNs;
  a.k_release = W + fault.extra;
  const unsigned hy = std::min(a.Hkv, kF32GridY), hz = (static_cast<unsigned>(a.Hkv) + kF32GridY - 1) / kF32GridY;
  const size_t smem = ns > 1 ? smem_for<D>(W, k) : F32Layout<D>::bytes(W);
  return launch_overlapped(attention_f32_kernel<D>, dim3(static_cast<unsigned>(a.Bt) * rb * ns, hy, hz),
                           dim3(32 * (W + 1)), smem, stream, static_cast<unsigned>(ns), a, rb, ns);
}

}  // namespace

cudaError_t launch_attention_f32(const AttnF32Args& a, cudaStream_t stream, const WaitFault& fault) {
  return a.d == 64 ? launch<64>(a, stream, fault) : launch<128>(a, stream, fault);
}

}  // namespace simsd
