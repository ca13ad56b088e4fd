// attention_tc64.cu -- bf16 verification attention for row blocks of at most
// 64 query rows on the sm_103a tensor cores (Sec. 3.2 "Target Model
// Verification", Sec. 3.3 KV cache): 8 drafts with 32/8 heads, 16 with 16/8.
//
// The same work units, split and merge as attention_tc.cu.  There a tile's
// S = Q K^T, softmax and O += P V follow one another (S has one TMEM buffer,
// since Q, S and O of 128 rows fill a CTA's 256 columns): 1.2 us a tile, of
// which the tensor core works 0.3.  That is enough where two CTAs an SM keep
// the memory busy, but a small batch has 2 to 24 tiles a CTA and waits for
// exactly this chain.  With 64 rows Q stays in shared memory (16 KB; the MMAs
// run over 128 rows, of which the upper 64 hold whatever lies behind Q and are
// never read), its TMEM columns become a second S buffer, and S of tile i+1 is
// computed while the softmax works on tile i: 0.5 to 0.9 us a tile.  Before ->
// now: 32 sequences of 4096 keys, 8 drafts 86.1 -> 82.0 us (547 MB, 98% of the
// copy rate); 19 of 190 to 3000 keys on 16-key pages with RoPE 50.7 -> 38.9;
// 36 layers of 8 sequences of 512 to 2048 784 -> 735.  The rest of a small
// batch's call is the first loads (2 to 4 us), the rotation (1.2), the split
// merge (3) and an uneven split of ragged prefixes.
//
// Warp roles (128 threads; two CTAs an SM, one warp of each on a scheduler):
//   warps 0-1  softmax; thread i owns query row i (TMEM lane i)
//   warp 2     TMA producer: Q, then K and V tiles of 16 KB in turn into a ring
//              of five slots; lane j issues the j-th box of a tile (two
//              d-halves of up to eight pages)
//   warp 3     MMA issuer (one thread) and TMEM owner
// TMEM (256 columns): S[2] [0,128) fp32 with P (bf16) over the first half of
// its buffer, O [128,256) fp32.
//
// Every mbarrier wait is bounded; a wait that expires sets SIMSD_EW_TIMEOUT
// and makes the whole CTA stop, drain its async work and free its TMEM.
#include <cooperative_groups.h>

#include <mutex>

#include "attention_tc.cuh"
#include "rope_tile.cuh"

namespace cg = cooperative_groups;

namespace simsd {
namespace {

constexpr int kThreads = 128;
constexpr int kWarpProducer = 2, kWarpMma = 3;
constexpr int kSoftmaxThreads = 64;
constexpr int kRopeThreads = 96;  // warps 0, 1 and the MMA warp
constexpr int kItems = 5;                    // ring slots: a K or a V tile each
constexpr int kItemBytes = 2 * kHalfBytes;   // two d-halves of 64 keys
constexpr int kQHalfBytes = kTc64Rows * 128;
constexpr uint32_t kTmemCols = 256, kColS = 0, kColO = 128;

struct alignas(1024) Smem64 {
  uint8_t q[2][kQHalfBytes];
  uint8_t ring[kItems][kItemBytes];
  uint64_t bar_q, bar_full[kItems], bar_free[kItems];
  uint64_t bar_s[2], bar_p[2], bar_pv[2], bar_drain;
  uint32_t tmem_base;
  int abort_flag;
  int seq_bad;
  int b_sel, n_sel;
  int32_t tau[64];
  int32_t pos[64];  // kRope: RoPE positions of the slots
  uint8_t sect[64];
  int32_t pages[kPageCache];
};

constexpr size_t smem_bytes() { return sizeof(Smem64) + 1024; }
static_assert(2 * (smem_bytes() + 1024) <= 233472, "two CTAs per SM");
static_assert((kPartWts + kRows / 2 * kWtsStride) * sizeof(float) <= sizeof(Smem64::q) + sizeof(Smem64::ring),
              "the fused split merge fits in Q and the ring");

__device__ __forceinline__ void signal_abort(Smem64& sm, int32_t* err_word) {
  raise_error(err_word, SIMSD_EW_TIMEOUT);
  *reinterpret_cast<volatile int*>(&sm.abort_flag) = 1;
}

// Item j of the ring (K of key tile j / 2 of this CTA when even, V when odd).
__device__ __forceinline__ uint32_t item_bar(const uint64_t* bars, uint32_t j) { return smem_u32(&bars[j % kItems]); }
__device__ __forceinline__ uint32_t item_phase(uint32_t j) { return (j / kItems) & 1; }

template <bool kFuse, bool kRope>
__global__ void __launch_bounds__(kThreads, 2)
    attention_tc64_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_kn,
                          const __grid_constant__ CUtensorMap tm_vn, const __grid_constant__ CUtensorMap tm_kc,
                          const __grid_constant__ CUtensorMap tm_vc, const __grid_constant__ TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  Smem64& sm =
      *reinterpret_cast<Smem64*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  volatile int* abort_flag = &sm.abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // which unit this CTA computes (as in attention_tc.cu)
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
    mbar_init(smem_u32(&sm.bar_q), 1);
    for (int i = 0; i < kItems; ++i) {
      mbar_init(smem_u32(&sm.bar_full[i]), 1);
      mbar_init(smem_u32(&sm.bar_free[i]), 1);
    }
    for (int u = 0; u < 2; ++u) {
      mbar_init(smem_u32(&sm.bar_s[u]), 1);
      mbar_init(smem_u32(&sm.bar_p[u]), 2 + p.extra_p);
      mbar_init(smem_u32(&sm.bar_pv[u]), 1);
    }
    mbar_init(smem_u32(&sm.bar_drain), 1);
    fence_mbar_init();
  }
  if (warp == kWarpMma) {
    tmem_alloc(smem_u32(&sm.tmem_base), kTmemCols);
    tmem_relinquish();
  }
  if (warp == kWarpProducer && lane == 0) {
    tma_prefetch_desc(&tm_q);
    tma_prefetch_desc(&tm_kn);
    tma_prefetch_desc(&tm_vn);
    tma_prefetch_desc(&tm_kc);
    tma_prefetch_desc(&tm_vc);
  }
  pdl_wait();
  // a CTA of a later wave lets the next kernel in at once, the others after
  // their tile loop (as in attention_tc.cu)
  if (static_cast<int>(blockIdx.x) >= p.slots) pdl_launch_next();
  __syncthreads();
  // several waves: sequences longest prefix first (ranked in the unused ring)
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
    fence_proxy_async_smem();  // the staging area is overwritten by TMA later
    __syncthreads();
    b = sm.b_sel;
    n = sm.n_sel;
  } else {
    b = rank;
  }
  const int32_t* bt = p.block_table + static_cast<size_t>(b) * p.max_pages;

  // One ring item of a key tile, by the producer warp (t = 0: the new slots,
  // t >= 1: prefix keys 64 (t - 1) ..): lane 0 announces the bytes, then lane
  // j issues box j (d-half j % 2 of page j / 2).
  auto issue_item = [&](uint32_t j, int t, int pi, int off) {
    const uint32_t bar = item_bar(sm.bar_full, j), dst = smem_u32(sm.ring[j % kItems]);
    const bool is_v = j & 1;
    const int half = lane & 1, sub = lane >> 1;
    if (t == 0) {
      if (lane == 0) mbar_arrive_expect_tx(bar, 2u * static_cast<uint32_t>(p.S) * 128u);
      __syncwarp();
      if (sub == 0) tma_load_3d(dst + half * kHalfBytes, is_v ? &tm_vn : &tm_kn, bar, 64 * half, kvh, b * p.S);
    } else {
      const int P = p.page_size, valid = min(kTile, n - (t - 1) * kTile);
      const int box = min(P, kTile), nsub = P >= kTile ? 1 : (valid + P - 1) / P;
      if (lane == 0) mbar_arrive_expect_tx(bar, 2u * static_cast<uint32_t>(nsub * box) * 128u);
      __syncwarp();
      if (sub < nsub) {
        const int pg = pi + sub < kPageCache ? sm.pages[pi + sub] : bt[pi + sub];
        tma_load_2d(dst + half * kHalfBytes + sub * box * 128, is_v ? &tm_vc : &tm_kc, bar, 64 * half,
                    (pg * p.Hkv + kvh) * P + off);
      }
    }
    __syncwarp();
  };
  // Q, and in split 0 the tile of new slots, need neither the prefix length
  // nor a page id: they go out first.  If the sequence turns out to be
  // invalid they are drained unused.
  uint32_t issued = 0;
  if (warp == kWarpProducer) {
    if (lane == 0) {
      const uint32_t bq = smem_u32(&sm.bar_q);
      const int qz = b * p.S + rblk * p.s_blk;
      mbar_arrive_expect_tx(bq, 2u * static_cast<uint32_t>(p.g * p.s_blk) * 128u);
      tma_load_3d(smem_u32(sm.q[0]), &tm_q, bq, 0, kvh * p.g, qz);
      tma_load_3d(smem_u32(sm.q[1]), &tm_q, bq, 64, kvh * p.g, qz);
    }
    __syncwarp();
    if (split == 0) {
      issue_item(0, 0, 0, 0);
      issue_item(1, 0, 0, 0);
      issued = 2;
    }
  }
  // The prefix length, the sequence's page ids (up to the page cache) and its
  // slot labels are read together: everything is in registers before the
  // first store, which the compiler must keep behind the loads before it.
  if (!p.sort) n = p.prefix_len[b];
  constexpr int kPgRegs = kPageCache / kThreads;
  int pg_reg[kPgRegs];
  const int pg_lim = min(p.max_pages, kPageCache);
#pragma unroll
  for (int j = 0; j < kPgRegs; ++j) {
    const int i = tid + j * kThreads;
    pg_reg[j] = i < pg_lim ? bt[i] : -1;
  }
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
    bool bad = false;
#pragma unroll
    for (int j = 0; j < kPgRegs; ++j) {
      const int i = tid + j * kThreads;
      if (i < npages) {
        sm.pages[i] = pg_reg[j];
        bad |= pg_reg[j] < 0 || pg_reg[j] >= p.num_pages;
      }
    }
    for (int i = kPageCache + tid; i < npages; i += kThreads) {
      const int pg = bt[i];
      bad |= pg < 0 || pg >= p.num_pages;
    }
    if (bad) {
      sm.seq_bad = 1;
      raise_error(p.err_word, SIMSD_EW_PAGE);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base;

  const bool seq_bad = sm.seq_bad != 0;
  const int T_all = seq_bad ? 0 : (n + kTile - 1) / kTile + 1;  // tile 0: new slots, 1..: prefix
  // the tiles of this split (as in attention_tc.cu: merged in a cluster,
  // split 0 holds tile 0, the costliest, and the fewest others)
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

  // Rotates this unit's queries and, in the split that holds them (its first
  // tile, ring items 0 and 1), the new keys at their slots' positions, by the
  // softmax warps and the MMA warp (ti: thread of 96).  A thread's first three
  // rounds of angles are formed while Q is in flight.
  auto rotate = [&](int ti, bool& ok) {
    constexpr int kStep = kRopeThreads / kRopeThreadsPerSlot, kAhead = 3;
    const bool keys_here = t0 == 0;
    const int q4 = ti % kRopeThreadsPerSlot;
    float2 f[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) f[e] = p.rope.f[4 * q4 + e];
    const int s0 = rblk * p.s_blk, s1 = min(p.S, s0 + p.s_blk);  // the slots of this block's query rows
    const int lo = (keys_here ? 0 : s0) + ti / kRopeThreadsPerSlot, hi = keys_here ? p.S : s1;
    float sn[kAhead][4], cs[kAhead][4];
#pragma unroll
    for (int r = 0; r < kAhead; ++r)
      if (lo + r * kStep < hi) rope_angles4(sm.pos[lo + r * kStep], f, sn[r], cs[r]);
    ok = mbar_wait_warp(smem_u32(&sm.bar_q), 0, abort_flag, p.wait_ns);
    if (ok && keys_here) ok = mbar_wait_warp(item_bar(sm.bar_full, 0), 0, abort_flag, p.wait_ns);
    if (ok) {
      auto turn = [&](int t, const float(&s)[4], const float(&c)[4]) {
        if (t >= s0 && t < s1) {
#pragma unroll 2
          for (int j = 0; j < p.g; ++j) rope_rotate4(sm.q[0], sm.q[1], (t - s0) * p.g + j, q4, s, c);
        }
        if (keys_here) rope_rotate4(sm.ring[0], sm.ring[0] + kHalfBytes, t, q4, s, c);
      };
#pragma unroll
      for (int r = 0; r < kAhead; ++r)
        if (lo + r * kStep < hi) turn(lo + r * kStep, sn[r], cs[r]);
#pragma unroll 1
      for (int t = lo + kAhead * kStep; t < hi; t += kStep) {
        rope_angles4(sm.pos[t], f, sn[0], cs[0]);
        turn(t, sn[0], cs[0]);
      }
      fence_proxy_async_smem();  // read next by the tensor core
    }
    asm volatile("bar.sync 1, 96;" ::: "memory");
  };

  // fused split merge: what the softmax thread of this row hands over
  bool fz_any = false, fz_have = false;
  float fz_m = -INFINITY, fz_l = 0.f;

  if (warp == kWarpProducer) {
    // ------------------------------------------------------------ producer
    bool ok = true;
    const int P = p.page_size;
    for (int i = 0; ok && i < ntiles; ++i) {
      const int t = t0 + i, key0 = max(0, t - 1) * kTile;
      const int pi = key0 / P, off = P >= kTile ? key0 - pi * P : 0;
      for (uint32_t j = 2 * i; ok && j < 2u * i + 2; ++j) {
        if (j < issued) continue;  // (the tile of new slots went out already)
        ok = j < kItems || mbar_wait_warp(item_bar(sm.bar_free, j), item_phase(j - kItems), abort_flag, p.wait_ns);
        if (!ok) break;
        issue_item(j, t, pi, off);
        issued = j + 1;
      }
    }
    if (lane == 0) {
      if (!ok) signal_abort(sm, p.err_word);
      // Drain: every issued load must have landed before the CTA may exit
      // (full limit, whatever the other waits use).
      mbar_wait(smem_u32(&sm.bar_q), 0, nullptr);
      for (uint32_t j = issued > kItems ? issued - kItems : 0; j < issued; ++j)
        mbar_wait(item_bar(sm.bar_full, j), item_phase(j), nullptr);
    }
    __syncwarp();
  } else if (warp == kWarpMma) {
    // ----------------------------------------------------------- MMA issuer
    bool ok = true;
    if (kRope && ntiles > 0) rotate(kSoftmaxThreads + lane, ok);
    if (lane == 0 && ntiles > 0) {
      constexpr uint32_t kIdescQK = idesc_bf16_f32(kRows, kTile, 0, 0);
      constexpr uint32_t kIdescPV = idesc_bf16_f32(kRows, kD, 0, 1);
      const uint32_t qb0 = smem_u32(sm.q[0]), qb1 = smem_u32(sm.q[1]);
      if (!kRope) ok = mbar_wait(smem_u32(&sm.bar_q), 0, abort_flag, p.wait_ns);
      // S of tile i needs K(i) and its buffer: PV(i - 2), which reads the P
      // in it, issued before (one thread's MMAs run in order).  PV of tile i
      // needs P(i) and V(i).  Whichever is ready goes next.
      int is = 0, iv = 0;
      unsigned long long t_idle = 0;
      for (uint32_t idle = 0; ok && iv < ntiles;) {
        bool moved = false;
        if (is < ntiles && is <= iv + 1 &&
            mbar_test_wait(item_bar(sm.bar_full, 2 * is), item_phase(2 * is))) {
          tc_fence_after();
          const uint32_t kb0 = smem_u32(sm.ring[(2 * is) % kItems]), kb1 = kb0 + kHalfBytes;
          const uint32_t scol = tmem + kColS + 64u * (is & 1);
#pragma unroll
          for (int kk = 0; kk < kD / 16; ++kk) {
            const uint32_t o = (kk & 3) * 32;
            tc_mma_ss(scol, sdesc_sw128((kk < 4 ? qb0 : qb1) + o, 16, 1024),
                      sdesc_sw128((kk < 4 ? kb0 : kb1) + o, 16, 1024), kIdescQK, kk > 0);
          }
          tc_commit(smem_u32(&sm.bar_s[is & 1]));
          tc_commit(item_bar(sm.bar_free, 2 * is));
          ++is;
          moved = true;
        }
        if (iv < is && mbar_test_wait(smem_u32(&sm.bar_p[iv & 1]), (iv >> 1) & 1) &&
            mbar_test_wait(item_bar(sm.bar_full, 2 * iv + 1), item_phase(2 * iv + 1))) {
          tc_fence_after();
          const uint32_t vb = smem_u32(sm.ring[(2 * iv + 1) % kItems]);
          const uint32_t pcol = tmem + kColS + 64u * (iv & 1);
#pragma unroll
          for (int kk = 0; kk < kTile / 16; ++kk)
            tc_mma_ts(tmem + kColO, pcol + 8 * kk, sdesc_sw128(vb + kk * 2048, kHalfBytes, 1024), kIdescPV,
                      (iv > 0 || kk > 0) ? 1u : 0u);
          tc_commit(smem_u32(&sm.bar_pv[iv & 1]));
          tc_commit(item_bar(sm.bar_free, 2 * iv + 1));
          ++iv;
          moved = true;
        }
        if (moved) {
          idle = 0;
        } else if ((++idle & 63u) == 0) {
          const unsigned long long now = globaltimer_ns();
          if (idle == 64) t_idle = now;
          if (*abort_flag || now - t_idle > p.wait_ns) ok = false;
        }
      }
      if (!ok) signal_abort(sm, p.err_word);
      // every MMA issued by this thread has completed once this fires
      tc_commit(smem_u32(&sm.bar_drain));
      mbar_wait(smem_u32(&sm.bar_drain), 0, nullptr);
    }
    __syncwarp();
  } else {
    // -------------------------------------------------------------- softmax
    const int row = tid;  // TMEM lane / query row
    const int s = rblk * p.s_blk + row / p.g;
    const int hl = row % p.g;
    const bool row_exists = row < p.rows_blk && s < p.S;
    const bool active = row_exists && !seq_bad && sm.sect[s] != kSectPad;
    const bool warp_rows = warp * 32 < p.rows_blk;  // (a block of up to 32 rows has none in warp 1)
    unsigned long long vis = slot_visibility(sm.tau, sm.sect, p.S, s);
    if (!active) vis = 0ull;
    const uint32_t lane_tmem = tmem + (static_cast<uint32_t>(warp * 32) << 16);
    float m_ref = -INFINITY, l_sum = 0.f;
    bool ok = true;
    if (kRope && ntiles > 0) rotate(tid, ok);

    for (int i = 0; ok && i < ntiles; ++i) {
      const int t = t0 + i;
      const uint32_t buf = i & 1, s_tmem = lane_tmem + kColS + 64u * buf;
      const bool is_new = t == 0;
      const int valid = is_new ? p.S : min(kTile, n - (t - 1) * kTile);
      if (warp_rows) {
        if (!mbar_wait_warp(smem_u32(&sm.bar_s[buf]), (i >> 1) & 1, abort_flag, p.wait_ns)) {
          ok = false;
          break;
        }
        tc_fence_after();
        uint32_t sa[32], sb[32];
        tmem_ld32(s_tmem, sa);
        tmem_ld32(s_tmem + 32, sb);
        tmem_wait_ld();
        float x[kTile];
#pragma unroll
        for (int c = 0; c < kTile; ++c) x[c] = __uint_as_float(c < 32 ? sa[c] : sb[c - 32]);
        if (is_new || valid < kTile) {
          // hide what the row may not see: one bit word per row and a select
          // per column (no divergence)
          const unsigned long long keep = is_new ? vis : ((1ull << valid) - 1ull);
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
          // O holds the earlier tiles: wait until the last PV has completed
          // (its barrier cannot pass another phase before this tile's P),
          // then scale it
          if (i > 0 &&
              !mbar_wait_warp(smem_u32(&sm.bar_pv[(i - 1) & 1]), ((i - 1) >> 1) & 1, abort_flag, p.wait_ns)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const float f = need ? fast_exp2(m_ref - mx) : 1.0f;
          if (need) {
            l_sum *= f;
            m_ref = mx;
          }
          if (i > 0) {
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
        }
        // p = 2^(s*scale*log2e - m): one FFMA and one MUFU.EX2 per score
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
        tmem_st32(s_tmem, pk);
        tmem_wait_st();
      } else if (i >= 2 &&
                 !mbar_wait_warp(smem_u32(&sm.bar_pv[buf]), ((i - 2) >> 1) & 1, abort_flag, p.wait_ns)) {
        // A warp without rows does not wait for S: it keeps its distance by
        // the PV two tiles back, so that neither its arrival for this tile
        // nor its wait for this V can be taken for an earlier phase's.
        ok = false;
        break;
      }
      if (valid < kTile || is_new) {
        // rows of V that no query may use are zeroed so that 0 * (stale or
        // non-finite data) cannot reach O
        const uint32_t jv = 2 * i + 1;
        if (!mbar_wait_warp(item_bar(sm.bar_full, jv), item_phase(jv), abort_flag, p.wait_ns)) {
          ok = false;
          break;
        }
        if (row >= valid || (is_new && sm.sect[row] == kSectPad)) {
          const uint4 z = make_uint4(0u, 0u, 0u, 0u);
          uint4* r0 = reinterpret_cast<uint4*>(sm.ring[jv % kItems] + row * 128);
          uint4* r1 = reinterpret_cast<uint4*>(sm.ring[jv % kItems] + kHalfBytes + row * 128);
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
      if (lane == 0) mbar_arrive(smem_u32(&sm.bar_p[buf]));
    }
    if (!ok && lane == 0) signal_abort(sm, p.err_word);
    pdl_launch_next();
    // ---- epilogue: O of the last PV (one thread's MMAs complete in order)
    const bool have_o = ok && ntiles > 0 &&
                        mbar_wait_warp(smem_u32(&sm.bar_pv[(ntiles - 1) & 1]), ((ntiles - 1) >> 1) & 1, abort_flag,
                                       p.wait_ns);
    if (have_o) tc_fence_after();
    const bool any = have_o && active && l_sum > 0.f;
    const int h = kvh * p.g + hl;
    if (kFuse) {
      // written to shared memory after the whole CTA is done with it (below)
      fz_any = any;
      fz_have = have_o;
      fz_m = m_ref;
      fz_l = l_sum;
    } else if (p.nsplit == 1) {
      const float inv = any ? 1.0f / l_sum : 0.f;
      // (a lane stores its own row: exchanging pieces first, as the partials
      // below do, made 32 x 4096 keys 82.1 -> 82.6 us)
      __nv_bfloat16* orow = p.out + ((static_cast<size_t>(b) * p.S + s) * p.Hq + h) * kD;
#pragma unroll 1
      for (int ch = 0; ch < kD / 32; ++ch) {
        uint32_t o[32];
        if (have_o) {
          tmem_ld32(lane_tmem + kColO + 32 * ch, o);
          tmem_wait_ld();
        }
        if (row_exists) {
          uint4 pkd[4];
          uint32_t* wv = reinterpret_cast<uint32_t*>(pkd);
#pragma unroll
          for (int c = 0; c < 16; ++c) {
            const float r0 = any ? __uint_as_float(o[2 * c]) * inv : 0.f;
            const float r1 = any ? __uint_as_float(o[2 * c + 1]) * inv : 0.f;
            wv[c] = pack_bf16x2(r0, r1);
          }
          uint4* dst = reinterpret_cast<uint4*>(orow + 32 * ch);
#pragma unroll
          for (int c = 0; c < 4; ++c) dst[c] = pkd[c];
        }
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
    // Merge of the splits of this unit: this CTA's partial O (unnormalised)
    // and (m, l) of each row go into Q and the ring, once every load and MMA
    // of the CTA has completed; then each CTA merges its share of the rows.
    cg::cluster_group cluster = cg::this_cluster();
    float* part = reinterpret_cast<float*>(sm.q[0]);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp < 2) {
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
    merge_unit(p, part, split, rblk, b, kvh);
    cluster_wait();  // no CTA leaves while a peer may still read its partials
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kWarpMma) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

}  // namespace

cudaError_t launch_attention_tc64(const CUtensorMap& tq, const CUtensorMap& tkn, const CUtensorMap& tvn,
                                  const CUtensorMap& tkc, const CUtensorMap& tvc, const TcParams& p,
                                  cudaStream_t stream) {
  {
    // the kernels' shared-memory attributes, once per device
    static std::mutex mu;
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(mu);
    if (!done[dev]) {
      for (auto kern : {attention_tc64_kernel<false, false>, attention_tc64_kernel<false, true>,
                        attention_tc64_kernel<true, false>, attention_tc64_kernel<true, true>}) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem_bytes()));
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
      }
      done[dev] = true;
    }
  }
  const long long grid = static_cast<long long>(p.Bt) * p.nsplit * p.Hkv * p.rb;
  auto kern = p.rope_pos ? (p.fuse ? attention_tc64_kernel<true, true> : attention_tc64_kernel<false, true>)
                         : (p.fuse ? attention_tc64_kernel<true, false> : attention_tc64_kernel<false, false>);
  return launch_overlapped(kern, dim3(static_cast<unsigned>(grid)), dim3(kThreads), smem_bytes(), stream,
                           p.fuse ? static_cast<unsigned>(p.nsplit) : 1u, tq, tkn, tvn, tkc, tvc, p);
}

}  // namespace simsd
