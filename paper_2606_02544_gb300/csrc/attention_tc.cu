// attention_tc.cu -- bf16 verification attention on the sm_103a tensor cores
// (row blocks of more than 64 query rows; up to 64 go to attention_tc64.cu)
// (Sec. 3.2 "Target Model Verification", Sec. 3.3 KV cache; the extra cost
// of the paired layout is linear in the prefix, Eqs. (4)-(5)).
//
// Work unit: (sequence b, KV head, row block, prefix split).  The query rows
// of one unit are the g = Hq/Hkv heads x 2*gamma slots that share the KV
// head ("GQA packing"), up to 128 rows, so QK^T and PV are M = 128 MMAs.
// Keys stream in tiles of 64: first one tile with the 2*gamma new slots, whose
// Eq. (1) visibility is evaluated on the fly from (section, tau), then the
// cached prefix pages (read through the page table with TMA).  When the
// inputs are not rotated yet (Sec. 3.1 RoPE copy), the softmax warps rotate
// Q and the new keys in shared memory before Q moves into TMEM and the first
// S is computed (rope_tile.cuh); cached keys are stored rotated.
//
// Two CTAs share each SM (96 KB of shared memory, 256 TMEM columns and 192
// threads apiece), so one CTA's set-up, first loads and epilogue overlap the
// other's streaming, and the two rings together keep the same bytes in
// flight as one large ring.
//
// Warp roles (192 threads):
//   warps 0-3  softmax; thread i owns query row i (TMEM lane i).  They first
//              move the Q tile from shared memory into TMEM, then per key
//              tile read S, update the running max / sum, write P (bf16)
//              over the first half of S and hand it to the MMA issuer.
//   warp 4     TMA producer (one thread): Q, then K/V tiles into a 3-deep
//              ring of 32 KB slots (Q uses the first slot once).
//   warp 5     MMA issuer (one thread) and TMEM owner.  Per tile:
//              S = Q K^T (TS MMA: Q in TMEM, K in shared memory) and, once P
//              is written, O += P V (TS MMA: P in TMEM, V MN-major in shared
//              memory).  The next S overwrites P, so it waits for that PV.
// TMEM (256 columns): Q [0,64) as bf16 pairs, S [64,128) fp32 with P in its
// first 32 columns, O [128,256) fp32.
//
// Every mbarrier wait is bounded; a wait that expires sets SIMSD_EW_TIMEOUT
// and makes the whole CTA stop, drain its async work and free its TMEM.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "attention_tc.cuh"
#include "rope_tile.cuh"

// Scratch of simsd_verify_attention_noalloc: the split partials live in this
// file-scope array instead of caller memory.  Every device that loads the
// library holds it until the process exits.  Host code must not use the
// symbol's address directly (on the host it is only a stand-in); it asks
// the runtime for the device address once per device (below).
static __device__ __align__(256) unsigned char g_noalloc_scratch[12u << 20];

namespace cg = cooperative_groups;

namespace simsd {
namespace {

constexpr int kStages = 3;           // ring slots of one CTA
constexpr int kThreads = 192;
constexpr int kCtasPerSm = 2;        // shared-memory budget of one CTA
// Registers per thread: at most 128, so that two CTAs fit one SM by the
// per-scheduler register file (each CTA's warps 0, 1, 4, 5 share two of the
// four schedulers).  With more, the block scheduler counts one CTA per SM: a
// launch still starts two per SM, but a freed slot is refilled only once its
// SM is empty, which left SMs idle for tens of microseconds on ragged
// prefixes.
constexpr int kMaxRegs = 128;
constexpr int kWarpProducer = 4;
constexpr int kWarpMma = 5;
constexpr uint32_t kTmemCols = 256;
constexpr uint32_t kColQ = 0, kColS = 64, kColO = 128;
constexpr int kSlotBytes = 4 * kHalfBytes;  // K0 K1 V0 V1, or Q0 Q1 (16 KB each)

struct alignas(1024) Smem {
  uint8_t ring[kStages][kSlotBytes];
  uint64_t bar_k[kStages], bar_v[kStages], bar_empty[kStages];
  uint64_t bar_qt, bar_s_full, bar_p, bar_pv, bar_drain;
  uint32_t tmem_base;
  int abort_flag;
  int seq_bad;
  int b_sel, n_sel;
  int32_t tau[64];
  int32_t pos[64];  // kRope: RoPE positions of the slots
  uint8_t sect[64];
  int32_t pages[kPageCache];
};

constexpr size_t smem_bytes() { return sizeof(Smem) + 1024; }
static_assert(kCtasPerSm * (smem_bytes() + 1024) <= 233472, "two CTAs per SM");
static_assert((kPartWts + kRows / 2 * kWtsStride) * sizeof(float) <= sizeof(Smem::ring),
              "the fused split merge fits in the ring");

__device__ __forceinline__ void signal_abort(Smem& sm, int32_t* err_word) {
  raise_error(err_word, SIMSD_EW_TIMEOUT);
  *reinterpret_cast<volatile int*>(&sm.abort_flag) = 1;
}

// Row r of a 128-byte-swizzled tile: 16-byte chunk c sits at chunk c ^ (r & 7).
__device__ __forceinline__ uint4 ld_sw128_chunk(const uint8_t* half, int r, int c) {
  return *reinterpret_cast<const uint4*>(half + r * 128 + ((c ^ (r & 7)) << 4));
}

// kFuse: the prefix splits of a unit form a cluster and merge their partials
// in shared memory (a separate instantiation, so that the unclustered kernel
// carries no cluster barriers).  kRope: queries and new keys arrive unrotated
// (also a separate instantiation: the plain one carries none of that code).
template <bool kFuse, bool kRope>
__global__ void __maxnreg__(kMaxRegs)
    attention_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_kn,
                        const __grid_constant__ CUtensorMap tm_vn, const __grid_constant__ CUtensorMap tm_kc,
                        const __grid_constant__ CUtensorMap tm_vc, const __grid_constant__ TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  Smem& sm = *reinterpret_cast<Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  volatile int* abort_flag = &sm.abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // ---- which unit this CTA computes; sequences go longest prefix first.
  // Merged in place, the splits of a unit are adjacent (one cluster);
  // otherwise the splits of a sequence follow one another.
  const int per_seq = p.nsplit * p.Hkv * p.rb;
  const int rank = blockIdx.x / per_seq;
  int rem = blockIdx.x - rank * per_seq;
  int split;
  if (kFuse) {
    split = rem % p.nsplit;
    rem /= p.nsplit;
  } else {
    split = rem / (p.Hkv * p.rb);
    rem -= split * p.Hkv * p.rb;
  }
  const int kvh = rem / p.rb;
  const int rblk = rem - kvh * p.rb;

  if (tid == 0) {
    sm.abort_flag = 0;
    sm.seq_bad = 0;
    sm.b_sel = rank;
  }
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&sm.bar_k[s]), 1);
      mbar_init(smem_u32(&sm.bar_v[s]), 1);
      mbar_init(smem_u32(&sm.bar_empty[s]), 1);
    }
    mbar_init(smem_u32(&sm.bar_qt), 1);
    mbar_init(smem_u32(&sm.bar_s_full), 1);
    mbar_init(smem_u32(&sm.bar_p), 4 + p.extra_p);
    mbar_init(smem_u32(&sm.bar_pv), 1);
    mbar_init(smem_u32(&sm.bar_drain), 1);
    fence_mbar_init();
  }
  if (warp == kWarpMma) {
    tmem_alloc(smem_u32(&sm.tmem_base), kTmemCols);
    tmem_relinquish();
  }
  if (warp == kWarpProducer && lane == 0) {
    // the tensor maps are kernel parameters, not results of earlier work
    tma_prefetch_desc(&tm_q);
    tma_prefetch_desc(&tm_kn);
    tma_prefetch_desc(&tm_vn);
    tma_prefetch_desc(&tm_kc);
    tma_prefetch_desc(&tm_vc);
  }
  // the set-up above touches no global memory; from here on the previous
  // kernel's results are needed
  pdl_wait();
  // A CTA of a later wave lets the next kernel in at once: the next grid can
  // then fill the slots this grid's last wave leaves idle (consecutive
  // layers).  First-wave CTAs let it in after their tile loop (below), so
  // that in a single-wave grid no waiting CTA of the next kernel sits beside
  // this one for its whole run (that cost up to 30 us with 32 sequences of
  // 4096-token prefixes).
  if (static_cast<int>(blockIdx.x) >= p.slots) pdl_launch_next();
  // the barriers and flags set by thread 0 above must be in place before the
  // producer (another warp) issues its first load on them
  __syncthreads();
  // When the grid takes more than one wave, the sequences go longest prefix
  // first: the prefix lengths are staged in the (still unused) ring and
  // ranked.  In a single wave every CTA is resident at once and the order
  // does not matter, so the CTA reads its own sequence's length only.
  int b, n = 0;
  if (p.sort) {
    int32_t* nval = reinterpret_cast<int32_t*>(sm.ring[0]);
    for (int i = tid; i < p.Bt; i += kThreads) nval[i] = p.prefix_len[i];
    __syncthreads();
    for (int i = tid; i < p.Bt; i += kThreads) {
      const int ni = nval[i];
      int r = 0;
      for (int j = 0; j < p.Bt; ++j) {
        const int nj = nval[j];
        r += (nj > ni) || (nj == ni && j < i);
      }
      if (r == rank) {
        sm.b_sel = i;
        sm.n_sel = ni;
      }
    }
    // the staging area is overwritten by TMA later
    fence_proxy_async_smem();
    __syncthreads();
    b = sm.b_sel;
    n = sm.n_sel;
  } else {
    b = rank;
  }
  const int32_t* bt = p.block_table + static_cast<size_t>(b) * p.max_pages;

  // ---- TMA issue of ring items (producer thread only): item 0 is Q, item
  // i + 1 is the i-th key tile of this unit (tile 0: new slots, 1..T: prefix)
  auto issue_q = [&]() {
    const uint32_t q_bytes = 2u * static_cast<uint32_t>(p.g * p.s_blk) * 128u;
    const int qz = b * p.S + rblk * p.s_blk;
    const uint32_t q0 = smem_u32(sm.ring[0]);
    mbar_arrive_expect_tx(smem_u32(&sm.bar_k[0]), q_bytes);
    tma_load_3d(q0, &tm_q, smem_u32(&sm.bar_k[0]), 0, kvh * p.g, qz);
    tma_load_3d(q0 + 2 * kHalfBytes, &tm_q, smem_u32(&sm.bar_k[0]), 64, kvh * p.g, qz);
    mbar_arrive(smem_u32(&sm.bar_v[0]));  // keeps the two barriers of slot 0 in step
  };
  auto issue_tile = [&](int it, int t) {
    const int P = p.page_size;
    const int st = it % kStages;
    const uint32_t bk = smem_u32(&sm.bar_k[st]), bv = smem_u32(&sm.bar_v[st]);
    const uint32_t k0 = smem_u32(sm.ring[st]), k1 = k0 + kHalfBytes;
    const uint32_t v0 = k0 + 2 * kHalfBytes, v1 = k0 + 3 * kHalfBytes;
    if (t > 0) {
      const int key0 = (t - 1) * kTile;
      const int valid = min(kTile, n - key0);
      if (P >= kTile) {
        const int pi = key0 / P;
        const int pg = pi < kPageCache ? sm.pages[pi] : bt[pi];
        const int row = (pg * p.Hkv + kvh) * P + (key0 % P);
        mbar_arrive_expect_tx(bk, 2u * kHalfBytes);
        tma_load_2d(k0, &tm_kc, bk, 0, row);
        tma_load_2d(k1, &tm_kc, bk, 64, row);
        mbar_arrive_expect_tx(bv, 2u * kHalfBytes);
        tma_load_2d(v0, &tm_vc, bv, 0, row);
        tma_load_2d(v1, &tm_vc, bv, 64, row);
      } else {
        const int nsub = (valid + P - 1) / P;
        const uint32_t sub_bytes = static_cast<uint32_t>(P) * 128u;
        mbar_arrive_expect_tx(bk, 2u * nsub * sub_bytes);
        for (int sb = 0; sb < nsub; ++sb) {
          const int pi = (key0 + sb * P) / P;
          const int pg = pi < kPageCache ? sm.pages[pi] : bt[pi];
          const int row = (pg * p.Hkv + kvh) * P;
          tma_load_2d(k0 + sb * sub_bytes, &tm_kc, bk, 0, row);
          tma_load_2d(k1 + sb * sub_bytes, &tm_kc, bk, 64, row);
        }
        mbar_arrive_expect_tx(bv, 2u * nsub * sub_bytes);
        for (int sb = 0; sb < nsub; ++sb) {
          const int pi = (key0 + sb * P) / P;
          const int pg = pi < kPageCache ? sm.pages[pi] : bt[pi];
          const int row = (pg * p.Hkv + kvh) * P;
          tma_load_2d(v0 + sb * sub_bytes, &tm_vc, bv, 0, row);
          tma_load_2d(v1 + sb * sub_bytes, &tm_vc, bv, 64, row);
        }
      }
    } else {
      const uint32_t new_bytes = static_cast<uint32_t>(p.S) * 128u;
      mbar_arrive_expect_tx(bk, 2u * new_bytes);
      tma_load_3d(k0, &tm_kn, bk, 0, kvh, b * p.S);
      tma_load_3d(k1, &tm_kn, bk, 64, kvh, b * p.S);
      mbar_arrive_expect_tx(bv, 2u * new_bytes);
      tma_load_3d(v0, &tm_vn, bv, 0, kvh, b * p.S);
      tma_load_3d(v1, &tm_vn, bv, 64, kvh, b * p.S);
    }
  };
  // Q, and in split 0 the tile of new slots, need neither the prefix length
  // nor a page id: they go out first.  If the sequence turns out to be
  // invalid they are drained unused.
  int early = 0;
  if (warp == kWarpProducer && lane == 0) {
    issue_q();
    early = 1;
    if (split == 0) {
      issue_tile(1, 0);
      early = 2;
    }
  }
  // The prefix length, the sequence's page ids (up to the page cache) and
  // its slot labels are read together: one memory latency instead of a
  // chain.  Page ids past the prefix are loaded but not used.
  if (!p.sort) n = p.prefix_len[b];
  constexpr int kPgRegs = (kPageCache + kThreads - 1) / kThreads;
  int pg_reg[kPgRegs];
  const int pg_lim = min(p.max_pages, kPageCache);
#pragma unroll
  for (int j = 0; j < kPgRegs; ++j) {
    const int i = tid + j * kThreads;
    pg_reg[j] = i < pg_lim ? bt[i] : -1;
  }
  // (S <= 64 slots, one a thread; everything is in registers before the
  // first store, which the compiler must keep behind the loads before it)
  int lab_t = 0, lab_pos = 0;
  uint8_t lab_s = 0;
  if (tid < p.S) {
    const size_t o = static_cast<size_t>(b) * p.S + tid;
    lab_t = p.tau[o];
    lab_s = p.section[o];
    if (kRope) lab_pos = p.rope_pos[o];
  }
  if (tid < p.S) {
    sm.tau[tid] = lab_t;
    sm.sect[tid] = lab_s;
    if (kRope) sm.pos[tid] = lab_pos;
  }
  const bool n_bad = n < 0 || static_cast<long long>(n) > static_cast<long long>(p.max_pages) * p.page_size;
  if (n_bad) {
    if (tid == 0) {
      sm.seq_bad = 1;
      raise_error(p.err_word, SIMSD_EW_PREFIX_LEN);
    }
  } else {
    const int npages = (n + p.page_size - 1) / p.page_size;
#pragma unroll
    for (int j = 0; j < kPgRegs; ++j) {
      const int i = tid + j * kThreads;
      if (i < npages && i < kPageCache) {
        const int pg = pg_reg[j];
        sm.pages[i] = pg;
        if (pg < 0 || pg >= p.num_pages) {
          sm.seq_bad = 1;
          raise_error(p.err_word, SIMSD_EW_PAGE);
        }
      }
    }
    for (int i = kPageCache + tid; i < npages; i += kThreads) {
      const int pg = bt[i];
      if (pg < 0 || pg >= p.num_pages) {
        sm.seq_bad = 1;
        raise_error(p.err_word, SIMSD_EW_PAGE);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base;

  const bool seq_bad = sm.seq_bad != 0;
  const int T = seq_bad ? 0 : (n + kTile - 1) / kTile;  // prefix tiles
  const int T_all = seq_bad ? 0 : T + 1;                 // tile 0: new slots, tiles 1..T: prefix
  // Split 0 always holds tile 0 (issued above).  Split i takes tiles
  // [ceil(i T_all / nsplit), ceil((i + 1) T_all / nsplit)); merged in a
  // cluster, where the slowest split sets the pace, split 0 instead holds
  // tile 0, the costliest (the Eq. (1) mask, zeroed V rows), plus tiles up
  // to floor(T_all / nsplit) in all, and splits 1.. share the rest evenly,
  // so the extra tiles of an uneven split go to splits without tile 0.
  int t0, t1;
  if (kFuse) {
    const int first = T_all == 0 ? 0 : max(1, T_all / p.nsplit);
    t0 = 0;
    t1 = first;
    if (split > 0) {
      const long long rest = T_all - first, ns1 = p.nsplit - 1;
      t0 = first + static_cast<int>(((split - 1) * rest + ns1 - 1) / ns1);
      t1 = first + static_cast<int>((split * rest + ns1 - 1) / ns1);
    }
  } else {
    t0 = static_cast<int>((static_cast<long long>(split) * T_all + p.nsplit - 1) / p.nsplit);
    t1 = static_cast<int>((static_cast<long long>(split + 1) * T_all + p.nsplit - 1) / p.nsplit);
  }
  const int ntiles = t1 - t0;

  // fused split merge: what the softmax thread of this row hands over
  bool fz_any = false, fz_have = false;
  float fz_m = -INFINITY, fz_l = 0.f;

  if (warp == kWarpProducer) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      int issued = early;
      if (ntiles > 0) {
        // Q (and in split 0 the tile of new slots) went out already
        for (int i = issued - 1; i < ntiles; ++i) {
          const int it = i + 1, st = it % kStages;
          if (it >= kStages &&
              !mbar_wait(smem_u32(&sm.bar_empty[st]), ((it / kStages) - 1) & 1, abort_flag, p.wait_ns)) {
            signal_abort(sm, p.err_word);
            break;
          }
          issue_tile(it, t0 + i);
          ++issued;
        }
      }
      // Drain: every issued load must have landed before the CTA may exit.
      // In a normal run these phases completed long ago.  These waits keep
      // the full limit even when a test shortens the others.
      for (int it = max(0, issued - kStages); it < issued; ++it) {
        const int st = it % kStages;
        mbar_wait(smem_u32(&sm.bar_k[st]), (it / kStages) & 1, nullptr);
        mbar_wait(smem_u32(&sm.bar_v[st]), (it / kStages) & 1, nullptr);
      }
    }
    __syncwarp();
  } else if (warp == kWarpMma) {
    // ----------------------------------------------------------- MMA issuer
    if (lane == 0 && ntiles > 0) {
      constexpr uint32_t kIdescQK = idesc_bf16_f32(kRows, kTile, 0, 0);
      constexpr uint32_t kIdescPV = idesc_bf16_f32(kRows, kD, 0, 1);
      auto issue_s = [&](int it) {
        const uint32_t kb0 = smem_u32(sm.ring[it % kStages]), kb1 = kb0 + kHalfBytes;
#pragma unroll
        for (int kk = 0; kk < kD / 16; ++kk) {
          const uint32_t ka = (kk < 4 ? kb0 : kb1) + (kk & 3) * 32;
          tc_mma_ts(tmem + kColS, tmem + kColQ + 8 * kk, sdesc_sw128(ka, 16, 1024), kIdescQK, kk > 0);
        }
        tc_commit(smem_u32(&sm.bar_s_full));
      };
      bool ok = mbar_wait(smem_u32(&sm.bar_qt), 0, abort_flag, p.wait_ns);
      bool s_issued = false;
      for (int i = 0; ok && i < ntiles; ++i) {
        const int it = i + 1, st = it % kStages;
        const uint32_t par = (it / kStages) & 1;
        // S overwrites P of the previous tile; tcgen05.mma ops issued by one
        // thread run in issue order, so that PV has read P before this S lands
        if (!s_issued) {
          if (!mbar_wait(smem_u32(&sm.bar_k[st]), par, abort_flag, p.wait_ns)) {
            ok = false;
            break;
          }
          tc_fence_after();
          issue_s(it);
        }
        s_issued = false;
        // V first: it has usually landed while the softmax works, and P is
        // then acted on at once (a tile's chain of S, softmax and PV is serial
        // within a CTA, 1.2 us of which the tensor core works 0.3; waiting in
        // this order and issuing the next S ahead of the commits: 64
        // sequences of 2048 to 8192 keys, 16 drafts 213.9 -> 204.2 us)
        if (!mbar_wait(smem_u32(&sm.bar_v[st]), par, abort_flag, p.wait_ns) ||
            !mbar_wait(smem_u32(&sm.bar_p), i & 1, abort_flag, p.wait_ns)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t vb = smem_u32(sm.ring[st]) + 2 * kHalfBytes;
#pragma unroll
        for (int kk = 0; kk < kTile / 16; ++kk) {
          tc_mma_ts(tmem + kColO, tmem + kColS + 8 * kk, sdesc_sw128(vb + kk * 2048, kHalfBytes, 1024),
                    kIdescPV, (i > 0 || kk > 0) ? 1u : 0u);
        }
        // the next tile's S goes right behind this PV when its K is there
        // (ahead of the commits, each of which holds the thread a while)
        if (i + 1 < ntiles && mbar_test_wait(smem_u32(&sm.bar_k[(it + 1) % kStages]), ((it + 1) / kStages) & 1)) {
          tc_fence_after();
          issue_s(it + 1);
          s_issued = true;
        }
        tc_commit(smem_u32(&sm.bar_empty[st]));
      }
      // The epilogue's barrier, committed once, behind the last PV.  (One
      // phase a tile would leave its wait ambiguous: S of the last tile is
      // handed over ahead of the commits of the PV before it, so a parity test
      // could find that PV's phase still open and take an older one for its
      // own.)
      if (ok) tc_commit(smem_u32(&sm.bar_pv));
      if (!ok) signal_abort(sm, p.err_word);
      // every MMA issued by this thread has completed once this fires
      tc_commit(smem_u32(&sm.bar_drain));
      mbar_wait(smem_u32(&sm.bar_drain), 0, nullptr);
    }
    __syncwarp();
  } else {
    // -------------------------------------------------------------- softmax
    const int row = tid;                       // TMEM lane / query row
    const int s = rblk * p.s_blk + row / p.g;
    const int hl = row % p.g;
    const bool row_exists = row < p.rows_blk && s < p.S;
    const bool active = row_exists && !seq_bad && sm.sect[s] != kSectPad;
    unsigned long long vis = slot_visibility(sm.tau, sm.sect, p.S, s);
    if (!active) vis = 0ull;
    const uint32_t lane_tmem = tmem + (static_cast<uint32_t>(warp * 32) << 16);
    float m_ref = -INFINITY, l_sum = 0.f;
    bool ok = true;

    // ---- Q: shared memory (ring slot 0) -> TMEM columns [0, 64)
    if (ntiles > 0) {
      if (!kRope) {
        ok = mbar_wait_warp(smem_u32(&sm.bar_k[0]), 0, abort_flag, p.wait_ns);
      } else {
        // rotate this unit's queries and, in the split that holds them (its
        // first tile, ring item 1), the new keys at their slots' positions;
        // a thread's first angles are formed while Q is in flight
        constexpr int st1 = 1 % kStages, kStep = 128 / kRopeThreadsPerSlot;
        const bool keys_here = t0 == 0;
        const int q4 = tid % kRopeThreadsPerSlot;
        float2 f[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) f[e] = p.rope.f[4 * q4 + e];
        const int s0 = rblk * p.s_blk, s1 = min(p.S, s0 + p.s_blk);  // the slots of this block's query rows
        const int lo = keys_here ? 0 : s0, hi = keys_here ? p.S : s1;
        int t = lo + tid / kRopeThreadsPerSlot;
        float sn[4], cs[4];
        if (t < hi) rope_angles4(sm.pos[t], f, sn, cs);
        ok = mbar_wait_warp(smem_u32(&sm.bar_k[0]), 0, abort_flag, p.wait_ns);
        if (ok && keys_here) ok = mbar_wait_warp(smem_u32(&sm.bar_k[st1]), 0, abort_flag, p.wait_ns);
        if (ok) {
#pragma unroll 1
          while (t < hi) {
            if (t >= s0 && t < s1) {
#pragma unroll 2
              for (int j = 0; j < p.g; ++j)
                rope_rotate4(sm.ring[0], sm.ring[0] + 2 * kHalfBytes, (t - s0) * p.g + j, q4, sn, cs);
            }
            if (keys_here) rope_rotate4(sm.ring[st1], sm.ring[st1] + kHalfBytes, t, q4, sn, cs);
            t += kStep;
            if (t < hi) rope_angles4(sm.pos[t], f, sn, cs);
          }
          // read next by the tensor core (keys) and overwritten by TMA (the
          // queries' slot)
          fence_proxy_async_smem();
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
      }
      if (ok) {
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          const uint8_t* half = sm.ring[0] + h * 2 * kHalfBytes;
          uint32_t qr[32];
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const uint4 v = ld_sw128_chunk(half, row, c);
            qr[4 * c] = v.x;
            qr[4 * c + 1] = v.y;
            qr[4 * c + 2] = v.z;
            qr[4 * c + 3] = v.w;
          }
          tmem_st32(lane_tmem + kColQ + 32 * h, qr);
        }
        tmem_wait_st();
      }
      tc_fence_before();
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (tid == 0 && ok && !*abort_flag) {
        mbar_arrive(smem_u32(&sm.bar_qt));
        mbar_arrive(smem_u32(&sm.bar_empty[0]));
      }
    }

    for (int i = 0; ok && i < ntiles; ++i) {
      const int it = i + 1, st = it % kStages;
      const int t = t0 + i;
      if (!mbar_wait_warp(smem_u32(&sm.bar_s_full), i & 1, abort_flag, p.wait_ns)) {
        ok = false;
        break;
      }
      tc_fence_after();
      uint32_t sa[32], sb[32];
      tmem_ld32(lane_tmem + kColS, sa);
      tmem_ld32(lane_tmem + kColS + 32, sb);
      tmem_wait_ld();

      const bool is_new = (t == 0);
      const int valid = is_new ? p.S : min(kTile, n - (t - 1) * kTile);
      float x[kTile];
#pragma unroll
      for (int c = 0; c < kTile; ++c) x[c] = __uint_as_float(c < 32 ? sa[c] : sb[c - 32]);
      if (is_new || valid < kTile) {
        // partial prefix tile or the tile of new slots: hide what the row may
        // not see.  One bit word per row and a select per column: the rows of
        // a warp see different new slots, so a per-column branch would
        // diverge (it cost microseconds on the first tile).
        const unsigned long long keep = is_new ? vis : (valid >= kTile ? ~0ull : ((1ull << valid) - 1ull));
        const uint32_t klo = static_cast<uint32_t>(keep), khi = static_cast<uint32_t>(keep >> 32);
#pragma unroll
        for (int c = 0; c < kTile; ++c) {
          const uint32_t bit = ((c < 32 ? klo : khi) >> (c & 31)) & 1u;
          x[c] = bit ? x[c] : -INFINITY;
        }
      }
      // raw-score maximum (pairwise tree); scale_log2 > 0 commutes with max
      float mx;
      {
        float r[kTile / 2];
#pragma unroll
        for (int c = 0; c < kTile / 2; ++c) r[c] = fmaxf(x[2 * c], x[2 * c + 1]);
#pragma unroll
        for (int w2 = kTile / 4; w2 >= 1; w2 >>= 1)
#pragma unroll
          for (int c = 0; c < w2; ++c) r[c] = fmaxf(r[c], r[c + w2]);
        mx = active ? r[0] * p.scale_log2 : -INFINITY;
      }
      bool need = false;
      if (active && mx != -INFINITY) {
        if (m_ref == -INFINITY)
          m_ref = mx;
        else if (mx > m_ref + kRescaleThreshold)
          need = true;
      }
      if (__any_sync(0xffffffffu, need)) {
        // O holds the earlier tiles; their PVs completed before this S was
        // computed (the S MMA waited for the last one)
        const float f = need ? fast_exp2(m_ref - mx) : 1.0f;
        if (need) {
          l_sum *= f;
          m_ref = mx;
        }
#pragma unroll 1
        for (int ch = 0; ch < kD / 32; ++ch) {
          uint32_t o[32];
          tmem_ld32(lane_tmem + kColO + 32 * ch, o);
          tmem_wait_ld();
#pragma unroll
          for (int c = 0; c < 32; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * f);
          tmem_st32(lane_tmem + kColO + 32 * ch, o);
        }
      }
      // p = 2^(s*scale*log2e - m): one FFMA and one MUFU.EX2 per score.  Rows
      // that are not active leave garbage in their own P/O rows only (MMA rows
      // are independent) and write zeros at the end.
      const float neg_m = (active && m_ref != -INFINITY) ? -m_ref : 0.f;
      uint32_t pk[32];
      float ps[kTile / 2];
#pragma unroll
      for (int c = 0; c < kTile / 2; ++c) {
        const float p0 = fast_exp2(fmaf(x[2 * c], p.scale_log2, neg_m));
        const float p1 = fast_exp2(fmaf(x[2 * c + 1], p.scale_log2, neg_m));
        ps[c] = p0 + p1;
        pk[c] = pack_bf16x2(p0, p1);
      }
#pragma unroll
      for (int w2 = kTile / 4; w2 >= 1; w2 >>= 1)
#pragma unroll
        for (int c = 0; c < w2; ++c) ps[c] += ps[c + w2];
      l_sum += ps[0];
      tmem_st32(lane_tmem + kColS, pk);
      tmem_wait_st();
      if (warp < 2 && (valid < kTile || is_new)) {
        // rows of V that no query may use are zeroed so that 0 * (stale or
        // non-finite data) cannot reach O
        if (!mbar_wait_warp(smem_u32(&sm.bar_v[st]), (it / kStages) & 1, abort_flag, p.wait_ns)) {
          ok = false;
          break;
        }
        const int kr = row;
        const bool zero = kr >= valid || (is_new && sm.sect[kr] == kSectPad);
        if (zero) {
          const uint4 z = make_uint4(0u, 0u, 0u, 0u);
          uint4* r0 = reinterpret_cast<uint4*>(sm.ring[st] + 2 * kHalfBytes + kr * 128);
          uint4* r1 = reinterpret_cast<uint4*>(sm.ring[st] + 3 * kHalfBytes + kr * 128);
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            r0[c] = z;
            r1[c] = z;
          }
        }
        fence_proxy_async_smem();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&sm.bar_p));
    }
    if (!ok && lane == 0) signal_abort(sm, p.err_word);
    // the next kernel on the stream may be scheduled now (its CTAs wait for
    // this grid to finish anyway); a clustered grid too, ahead of its merge:
    // the next layer's set-up then runs under it (36 layers of 8 sequences of
    // 512 to 2048 keys, 16 drafts: 734 us with the trigger at exit, 703 here)
    pdl_launch_next();
    // ---- epilogue: O of the last PV, scaled by 1/l (bar_pv has one phase: it
    // completes when every MMA of the CTA has)
    const bool have_o = ok && ntiles > 0 && mbar_wait_warp(smem_u32(&sm.bar_pv), 0, abort_flag, p.wait_ns);
    if (have_o) tc_fence_after();
    const bool any = have_o && active && l_sum > 0.f;
    const int h = kvh * p.g + hl;
    if (kFuse) {
      // written to the ring after the whole CTA is done with it (below)
      fz_any = any;
      fz_have = have_o;
      fz_m = m_ref;
      fz_l = l_sum;
    } else if (p.nsplit == 1) {
      const float inv = any ? 1.0f / l_sum : 0.f;
      const int at = row_exists ? (b * p.S + s) * p.Hq + h : -1;
#pragma unroll 1
      for (int ch = 0; ch < kD / 32; ++ch) {
        uint32_t o[32];
        if (have_o) {
          tmem_ld32(lane_tmem + kColO + 32 * ch, o);
          tmem_wait_ld();
        }
        store_chunk_bf16(o, any, inv, p.out, at, ch);
      }
    } else {
      const size_t unit = ((static_cast<size_t>(b) * p.Hkv + kvh) * p.rb + rblk) * p.nsplit + split;
      const size_t nunits = static_cast<size_t>(p.Bt) * p.Hkv * p.rb * p.nsplit;
      float* wo = p.ws + unit * p.rows_blk * kD;
      float* wml = p.ws + nunits * p.rows_blk * kD + (unit * p.rows_blk + row) * 2;
      const int at = row < p.rows_blk ? row : -1;
#pragma unroll 1
      for (int ch = 0; ch < kD / 32; ++ch) {
        uint32_t o[32];
        if (have_o) {
          tmem_ld32(lane_tmem + kColO + 32 * ch, o);
          tmem_wait_ld();
        }
        store_chunk_f32(o, any, wo, at, ch);
      }
      if (row < p.rows_blk) {
        wml[0] = any ? m_ref : -INFINITY;
        wml[1] = any ? l_sum : 0.f;
      }
    }
  }

  if (kFuse) {
    // Merge of the splits of this unit, O = sum_i 2^(m_i - M) O_i / sum_i
    // 2^(m_i - M) l_i: CTA c of the cluster takes rows c, c + nsplit, ...,
    // reading every split's partials through distributed shared memory.
    // First this CTA's partial O (unnormalised) and (m, l) of each row go
    // into the ring, once every load and MMA of the CTA has completed.
    cg::cluster_group cluster = cg::this_cluster();
    float* part = reinterpret_cast<float*>(sm.ring[0]);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp < 4) {
      const int row = tid;
      const uint32_t lane_tmem = tmem + (static_cast<uint32_t>(warp * 32) << 16);
#pragma unroll 1
      for (int ch = 0; ch < kD / 32; ++ch) {
        uint32_t o[32];
        if (fz_have) {
          tmem_ld32(lane_tmem + kColO + 32 * ch, o);
          tmem_wait_ld();
        }
        if (row < p.rows_blk) {
          float4* dst = reinterpret_cast<float4*>(part + row * kPartStride + 32 * ch);
#pragma unroll
          for (int c = 0; c < 8; ++c)
            dst[c] = fz_any ? make_float4(__uint_as_float(o[4 * c]), __uint_as_float(o[4 * c + 1]),
                                          __uint_as_float(o[4 * c + 2]), __uint_as_float(o[4 * c + 3]))
                            : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
      if (row < p.rows_blk) {
        part[kPartMl + 2 * row] = fz_any ? fz_m : -INFINITY;
        part[kPartMl + 2 * row + 1] = fz_any ? fz_l : 0.f;
      }
    }
    cluster.sync();  // every split's partials are in place
    if (warp < 4) {
      merge_unit(p, part, split, rblk, b, kvh);
    } else {
      cluster_arrive();
    }
    cluster_wait();  // no CTA leaves while a peer may still read its partials
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kWarpMma) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

// Merges the prefix splits of every (sequence, KV head, row block):
// O = sum_i 2^(m_i - M) O_i / sum_i 2^(m_i - M) l_i.  One warp per row; the
// lanes take the splits' (m, l) in parallel, then sum the partial O rows with
// lanes over the head dimension (independent loads, several in flight).
__global__ void __launch_bounds__(128) combine_kernel(const __grid_constant__ TcParams p) {
  constexpr int kBatch = 4;  // splits whose partials a lane loads before adding any
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const unsigned full = 0xffffffffu;
  const long long wid = (static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const long long units = static_cast<long long>(p.Bt) * p.Hkv * p.rb;
  if (wid >= units * p.rows_blk) return;
  const int row = static_cast<int>(wid % p.rows_blk);
  const long long u = wid / p.rows_blk;
  const int rblk = static_cast<int>(u % p.rb);
  const int kvh = static_cast<int>((u / p.rb) % p.Hkv);
  const int b = static_cast<int>(u / (static_cast<long long>(p.rb) * p.Hkv));
  const int s = rblk * p.s_blk + row / p.g;
  if (s >= p.S) return;
  const int h = kvh * p.g + row % p.g;
  const size_t nunits = static_cast<size_t>(units) * p.nsplit;
  const float* wml = p.ws + nunits * p.rows_blk * kD;
  const size_t e0 = static_cast<size_t>(u) * p.nsplit;
  float M = -INFINITY;
  for (int i = lane; i < p.nsplit; i += 32) {
    const size_t e = (e0 + i) * p.rows_blk + row;
    if (wml[2 * e + 1] > 0.f) M = fmaxf(M, wml[2 * e]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(full, M, o));
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  float L = 0.f;
  if (M != -INFINITY) {
    for (int c0 = 0; c0 < p.nsplit; c0 += 32) {
      // lane j holds the weight of split c0 + j
      float wj = 0.f;
      if (c0 + lane < p.nsplit) {
        const size_t e = (e0 + c0 + lane) * p.rows_blk + row;
        const float lj = wml[2 * e + 1];
        if (lj > 0.f) {
          wj = exp2f(wml[2 * e] - M);
          L = fmaf(wj, lj, L);
        }
      }
      const int cnt = min(32, p.nsplit - c0);
      // the partials of kBatch splits are loaded before any is added (one
      // round trip per batch; the sum keeps the split order)
      const float4* ob = reinterpret_cast<const float4*>(p.ws + ((e0 + c0) * p.rows_blk + row) * kD) + lane;
      const size_t split4 = static_cast<size_t>(p.rows_blk) * (kD / 4);  // float4s from one split to the next
      for (int j0 = 0; j0 < cnt; j0 += kBatch) {
        float4 o[kBatch];
#pragma unroll
        for (int j = 0; j < kBatch; ++j)
          o[j] = j0 + j < cnt ? ob[(j0 + j) * split4] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
          if (j0 + j < cnt) {  // (the same for the whole warp)
            const float w = __shfl_sync(full, wj, j0 + j);
            acc.x = fmaf(w, o[j].x, acc.x);
            acc.y = fmaf(w, o[j].y, acc.y);
            acc.z = fmaf(w, o[j].z, acc.z);
            acc.w = fmaf(w, o[j].w, acc.w);
          }
        }
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) L += __shfl_xor_sync(full, L, o);
  const float inv = L > 0.f ? 1.f / L : 0.f;
  __nv_bfloat16* orow = p.out + ((static_cast<size_t>(b) * p.S + s) * p.Hq + h) * kD;
  uint2 v;
  v.x = pack_bf16x2(acc.x * inv, acc.y * inv);
  v.y = pack_bf16x2(acc.z * inv, acc.w * inv);
  reinterpret_cast<uint2*>(orow)[lane] = v;
  // the next kernel is let in only as this grid's blocks finish: launched
  // at the start, its CTAs took SMs that thousands of these small blocks
  // still needed
  pdl_launch_next();
}

// The same for many splits of few rows: a block per row, its four warps taking
// the splits in turn (warp w: w, w + 4, ...; at most kRowPer each).  Every
// partial of the row and every (m, l) is requested at once, each warp folds
// its splits under its own maximum, and the four results are merged in shared
// memory: one round trip to memory.  A warp per row walked the (m, l) twice
// and the partials in batches of 16, four or five dependent round trips.
constexpr int kRowPer = 16;
__global__ void __launch_bounds__(128) combine_row_kernel(const __grid_constant__ TcParams p) {
  __shared__ float4 acc_s[4][32];
  __shared__ float m_s[4], l_s[4];
  pdl_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned full = 0xffffffffu;
  const int row = static_cast<int>(blockIdx.x % p.rows_blk);
  const unsigned u = blockIdx.x / p.rows_blk;
  const int rblk = static_cast<int>(u % p.rb);
  const int kvh = static_cast<int>((u / p.rb) % p.Hkv);
  const int b = static_cast<int>(u / (static_cast<unsigned>(p.rb) * p.Hkv));
  const int s = rblk * p.s_blk + row / p.g;
  if (s >= p.S) return;  // (the same for the whole block)
  const size_t units = static_cast<size_t>(p.Bt) * p.Hkv * p.rb, e0 = static_cast<size_t>(u) * p.nsplit;
  const float2* wml = reinterpret_cast<const float2*>(p.ws + units * p.nsplit * p.rows_blk * kD);
  const int cnt = (p.nsplit - warp + 3) / 4;  // this warp's splits
  // lane j: (m, l) of split warp + 4 j
  const float2 ml = lane < cnt ? wml[(e0 + warp + 4 * lane) * p.rows_blk + row] : make_float2(-INFINITY, 0.f);
  float4 x[kRowPer];
#pragma unroll
  for (int j = 0; j < kRowPer; ++j)
    x[j] = j < cnt ? reinterpret_cast<const float4*>(p.ws + ((e0 + warp + 4 * j) * p.rows_blk + row) * kD)[lane]
                   : make_float4(0.f, 0.f, 0.f, 0.f);
  float M = ml.y > 0.f ? ml.x : -INFINITY;
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(full, M, o));
  M = __shfl_sync(full, M, 0);
  const float w = ml.y > 0.f ? exp2f(ml.x - M) : 0.f;
  float L = w * ml.y;
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) L += __shfl_xor_sync(full, L, o);
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int j = 0; j < kRowPer; ++j) {
    const float wj = __shfl_sync(full, w, j);
    acc.x = fmaf(wj, x[j].x, acc.x);
    acc.y = fmaf(wj, x[j].y, acc.y);
    acc.z = fmaf(wj, x[j].z, acc.z);
    acc.w = fmaf(wj, x[j].w, acc.w);
  }
  acc_s[warp][lane] = acc;
  if (lane == 0) {
    m_s[warp] = M;
    l_s[warp] = L;
  }
  __syncthreads();
  if (warp == 0) {
    float Ma = m_s[0], La = 0.f;
#pragma unroll
    for (int k = 1; k < 4; ++k) Ma = fmaxf(Ma, m_s[k]);
    float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float f = l_s[k] > 0.f ? exp2f(m_s[k] - Ma) : 0.f;
      const float4 v = acc_s[k][lane];
      La = fmaf(f, l_s[k], La);
      y.x = fmaf(f, v.x, y.x);
      y.y = fmaf(f, v.y, y.y);
      y.z = fmaf(f, v.z, y.z);
      y.w = fmaf(f, v.w, y.w);
    }
    const float inv = La > 0.f ? 1.f / La : 0.f;
    const int h = kvh * p.g + row % p.g;
    reinterpret_cast<uint2*>(p.out + ((static_cast<size_t>(b) * p.S + s) * p.Hq + h) * kD)[lane] =
        make_uint2(pack_bf16x2(y.x * inv, y.y * inv), pack_bf16x2(y.z * inv, y.w * inv));
  }
  // (the next kernel is let in as this grid's blocks finish, as above)
  pdl_launch_next();
}

// The kernels' shared-memory attributes, set once per device (function
// attributes apply to the current device only).
cudaError_t ensure_smem_attr() {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(mu);
  if (done[dev]) return cudaSuccess;
  for (auto kern : {attention_tc_kernel<false, false>, attention_tc_kernel<false, true>,
                    attention_tc_kernel<true, false>, attention_tc_kernel<true, true>}) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem_bytes()));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  done[dev] = true;
  return cudaSuccess;
}

bool make_map(EncodeTiledFn encode, CUtensorMap* m, const void* base, int rank, const cuuint64_t* dims,
              const cuuint64_t* strides, const cuuint32_t* box) {
  return make_bf16_map(encode, m, base, rank, dims, strides, box);
}

}  // namespace

bool make_bf16_map(EncodeTiledFn encode, CUtensorMap* m, const void* base, int rank, const cuuint64_t* dims,
                   const cuuint64_t* strides, const cuuint32_t* box) {
  cuuint32_t es[3] = {1, 1, 1};
  return encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(base), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool plan_attention_tc(int Bt, int gamma, int Hq, int Hkv, int max_pages, int page_size, int num_sms,
                       AttnTcPlan* plan, bool allow_streamk) {
  const int S = 2 * gamma, g = Hq / Hkv;
  const int R = g * S;
  AttnTcPlan pl{};
  if (R <= kRows) {
    pl.rb = 1;
    pl.s_blk = S;
  } else {
    if (kRows % g != 0) return false;
    pl.s_blk = kRows / g;
    pl.rb = (S + pl.s_blk - 1) / pl.s_blk;
  }
  pl.rows_blk = g * pl.s_blk;
  if (pl.rows_blk > kRows || g > 256 || pl.s_blk > 256) return false;
  pl.num_sms = num_sms;
  const long long max_tiles = (static_cast<long long>(max_pages) * page_size + kTile - 1) / kTile + 1;
  if (const int ns256 = tc256_splits(Bt, Hkv, pl.rb, max_tiles, num_sms)) {
    // two row blocks share one CTA and its K/V stream; with fewer units
    // than SMs each unit's key tiles are split into ranges whose partials
    // the combine kernel merges
    pl.kind = 1;
    pl.streamk = allow_streamk ? tc256_streamk(Bt, Hkv, max_tiles, ns256, num_sms) : 0;
    pl.nsplit = pl.streamk ? 1 : ns256;
    pl.sort = 0;
    pl.fuse = 0;
    pl.slots = num_sms;
    pl.ws_bytes = pl.streamk ? tc256_streamk_bytes(num_sms)
                  : pl.nsplit > 1
                      ? static_cast<size_t>(Bt) * Hkv * pl.rb * pl.nsplit * pl.rows_blk * (kD + 2) * sizeof(float)
                      : 0;
    *plan = pl;
    return true;
  }
  // split the prefix only when the units alone cannot fill the GPU (the
  // occupancy calculator reports one CTA per SM for this kernel although two
  // are resident, so the budget the kernel is built for is used instead)
  const long long units = static_cast<long long>(Bt) * Hkv * pl.rb;
  const long long slots = static_cast<long long>(num_sms) * kCtasPerSm;
  int ns = 1;
  if (units < slots) {
    // as many splits as keep every CTA in one wave
    ns = static_cast<int>(std::max<long long>(1, slots / units));
    ns = static_cast<int>(std::min<long long>(ns, std::max<long long>(1, max_tiles / 2)));
    ns = std::min(ns, 64);
  }
  pl.nsplit = ns;
  pl.sort = (units * ns > slots && Bt <= 256) ? 1 : 0;
  // up to 8 splits merge in place (a cluster per unit), more through the
  // workspace and combine_kernel
  pl.fuse = (ns >= 2 && ns <= kMaxSplitFuse) ? 1 : 0;
  pl.slots = static_cast<int>(slots);
  pl.ws_bytes = (ns > 1 && !pl.fuse) ? static_cast<size_t>(units) * ns * pl.rows_blk * (kD + 2) * sizeof(float) : 0;
  *plan = pl;
  return true;
}

// The combine launch: a block per row for more than 4 splits of few rows (a
// small batch), a warp per row otherwise (a large grid merging a few splits a
// row needs its blocks resident more than loads in flight).  The whole call at
// one sequence, 38 splits of each row, a warp a row -> a block a row: 32768
// keys 35.4 -> 32.6 us, 8192 keys 18.4 -> 15.2 (31.7 and 13.7 by now).
cudaError_t launch_combine(const TcParams& p, long long rows, int num_sms, cudaStream_t stream) {
  if (p.nsplit > 4 && p.nsplit <= 4 * kRowPer && rows <= 16LL * num_sms)
    return launch_overlapped(combine_row_kernel, dim3(static_cast<unsigned>(rows)), dim3(128), 0, stream, 1, p);
  return launch_overlapped(combine_kernel, dim3(static_cast<unsigned>((rows + 3) / 4)), dim3(128), 0, stream, 1, p);
}

cudaError_t launch_attention_combine(const AttnTcArgs& a, const AttnTcPlan& pl, cudaStream_t stream) {
  TcParams p{};
  p.out = static_cast<__nv_bfloat16*>(a.out);
  p.ws = static_cast<float*>(a.workspace);
  p.Bt = a.Bt;
  p.gamma = a.gamma;
  p.S = 2 * a.gamma;
  p.Hq = a.Hq;
  p.Hkv = a.Hkv;
  p.g = a.Hq / a.Hkv;
  p.rb = pl.rb;
  p.rows_blk = pl.rows_blk;
  p.s_blk = pl.s_blk;
  p.nsplit = pl.nsplit;
  const long long warps = static_cast<long long>(a.Bt) * a.Hkv * pl.rb * pl.rows_blk;
  return launch_combine(p, warps, pl.num_sms, stream);
}

cudaError_t launch_attention_tc(const AttnTcArgs& a, const AttnTcPlan& pl, EncodeTiledFn encode,
                                cudaStream_t stream) {
  if (pl.kind == 1) return launch_attention_tc256(a, pl, encode, stream);
  const int S = 2 * a.gamma, g = a.Hq / a.Hkv;
  CUtensorMap tq, tkn, tvn, tkc, tvc;
  {
    const cuuint64_t dims[3] = {static_cast<cuuint64_t>(kD), static_cast<cuuint64_t>(a.Hq),
                                static_cast<cuuint64_t>(a.Bt) * S};
    const cuuint64_t strides[2] = {kD * 2ull, static_cast<cuuint64_t>(a.Hq) * kD * 2ull};
    const cuuint32_t box[3] = {64u, static_cast<cuuint32_t>(g), static_cast<cuuint32_t>(pl.s_blk)};
    if (!make_map(encode, &tq, a.q, 3, dims, strides, box)) return cudaErrorInvalidValue;
  }
  {
    const cuuint64_t dims[3] = {static_cast<cuuint64_t>(kD), static_cast<cuuint64_t>(a.Hkv),
                                static_cast<cuuint64_t>(a.Bt) * S};
    const cuuint64_t strides[2] = {kD * 2ull, static_cast<cuuint64_t>(a.Hkv) * kD * 2ull};
    const cuuint32_t box[3] = {64u, 1u, static_cast<cuuint32_t>(S)};
    if (!make_map(encode, &tkn, a.k_new, 3, dims, strides, box)) return cudaErrorInvalidValue;
    if (!make_map(encode, &tvn, a.v_new, 3, dims, strides, box)) return cudaErrorInvalidValue;
  }
  {
    // a pool without pages is described by a one-row map that is never read
    const cuuint64_t dims[2] = {static_cast<cuuint64_t>(kD),
                                std::max<cuuint64_t>(1, static_cast<cuuint64_t>(a.num_pages) * a.Hkv * a.page_size)};
    const cuuint64_t strides[1] = {kD * 2ull};
    const cuuint32_t box[2] = {64u, static_cast<cuuint32_t>(std::min(a.page_size, kTile))};
    if (!make_map(encode, &tkc, a.k_cache, 2, dims, strides, box)) return cudaErrorInvalidValue;
    if (!make_map(encode, &tvc, a.v_cache, 2, dims, strides, box)) return cudaErrorInvalidValue;
  }
  TcParams p{};
  p.block_table = a.block_table;
  p.prefix_len = a.prefix_len;
  p.tau = a.tau;
  p.section = a.section;
  p.rope_pos = a.rope_pos;
  p.rope = a.rope;
  p.out = static_cast<__nv_bfloat16*>(a.out);
  p.ws = static_cast<float*>(a.workspace);
  p.err_word = a.err_word;
  p.max_pages = a.max_pages;
  p.page_size = a.page_size;
  p.num_pages = a.num_pages;
  p.Bt = a.Bt;
  p.gamma = a.gamma;
  p.S = S;
  p.Hq = a.Hq;
  p.Hkv = a.Hkv;
  p.g = g;
  p.rb = pl.rb;
  p.rows_blk = pl.rows_blk;
  p.s_blk = pl.s_blk;
  p.nsplit = pl.nsplit;
  p.sort = pl.sort;
  p.fuse = pl.fuse;
  p.slots = pl.slots;
  p.scale_log2 = a.scale * 1.4426950408889634f;
  p.wait_ns = a.fault.wait_ns ? a.fault.wait_ns : kWaitLimitNs;
  p.extra_p = a.fault.extra;

  {
    cudaError_t e = ensure_smem_attr();
    if (e != cudaSuccess) return e;
  }
  const long long grid = static_cast<long long>(a.Bt) * pl.nsplit * a.Hkv * pl.rb;
  if (pl.rows_blk <= kTc64Rows) {
    cudaError_t e = launch_attention_tc64(tq, tkn, tvn, tkc, tvc, p, stream);
    if (e != cudaSuccess || pl.nsplit == 1 || pl.fuse) return e;
    return launch_combine(p, static_cast<long long>(a.Bt) * a.Hkv * pl.rb * pl.rows_blk, pl.num_sms, stream);
  }
  auto kern = a.rope_pos ? (pl.fuse ? attention_tc_kernel<true, true> : attention_tc_kernel<false, true>)
                         : (pl.fuse ? attention_tc_kernel<true, false> : attention_tc_kernel<false, false>);
  cudaError_t e = launch_overlapped(kern, dim3(static_cast<unsigned>(grid)), dim3(kThreads), smem_bytes(), stream,
                                    pl.fuse ? static_cast<unsigned>(pl.nsplit) : 1u, tq, tkn, tvn, tkc, tvc, p);
  if (e != cudaSuccess || pl.nsplit == 1 || pl.fuse) return e;
  const long long warps = static_cast<long long>(a.Bt) * a.Hkv * pl.rb * pl.rows_blk;
  return launch_combine(p, warps, pl.num_sms, stream);
}

size_t noalloc_scratch_capacity() { return sizeof(g_noalloc_scratch); }

cudaError_t noalloc_scratch_pointer(void** out) {
  // Set-up, once per device and with that device current: the device
  // address of the static scratch array.  It is kept for the life of the
  // process (a device reset, which would move the array, is not supported).
  static std::mutex mu;
  static void* ptr[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(mu);
  if (!ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    ptr[dev] = p;
  }
  *out = ptr[dev];
  return cudaSuccess;
}

}  // namespace simsd
