// Forward pass of block-sparse causal attention (paper Section 3.2: a FlashAttention-style
// kernel that never loads or computes a KV block whose mask is zero), with the log-sum-exp.
//
// One CTA owns a super-tile of 256 query rows of one head: two tiles ("slots") of 128 rows
// that share every K / V tile brought into shared memory.  It walks the ascending union of
// the slots' active KV blocks in steps of 128 keys (one 128-token block, or two 64-token
// blocks side by side), each step in two halves of 64 keys; a slot skips the halves none of
// its rows can see.  Roles:
//   warps 0-3 / 4-7 : softmax of slot 0 / 1 (thread = query row = TMEM lane)
//   warp 8          : TMA producer (Q once, then the K and V rings)
//   warps 9 / 10    : issue the tcgen05.mma of slot 0 / 1 (warp-uniform code, one elected lane;
//                     the two warps sit on different scheduler partitions of the SM)
// Tensor memory, D = 128: S of slot s, half h at columns 128 s + 64 h (P is written as bf16 over the
// first 32 of them), O of slot s at 256 + 128 s.  Per slot the issue order is
//   S_0(0) S_1(0) | PV_0(0) S_0(1) | PV_1(0) S_1(1) | PV_0(1) S_0(2) | ...
// so the two halves of a slot form a double buffer: while the softmax works on one half the
// tensor pipe computes the other, and the second slot fills what is left.
// D = 64: the products of a half take 320 cycles of the tensor pipe where its exponentials take 512 of
// the exponential unit, so the element-wise chain sets the pace, and what fills the unit is more rows in
// work.  Grids that fill the chip several times over (fwd_two_ctas, lg_host.h) therefore run two CTAs on an SM (NB = 1):
// each has half the tensor memory, one score buffer per slot (S of slot s at 64 s, O at 128 + 64 s;
// S(0) | PV(0) S(1) | PV(1) S(2) | ...) and 80 registers per thread, hence the half is worked 32 columns at a time (3 x 16 /
// 4 heads x 6001 tokens, window 1024: 164 -> 148 us with 64- and with 128-token blocks, although 13 / 34 registers are
// spilled there).  Both forms sum in the same order and give the same bits.
// Grids of few heads cut long super-tiles along their keys (fwd_split, lg_pattern.h): kSplit, a CTA per piece, a tile's in one
// cluster, which adds them (fwd_join).
// The online softmax advances half by half.  A row's reference (the maximum its probabilities are expressed relative
// to) only moves, and O is only rescaled, when a half's probabilities sum to more than 2^8;
// until then they are relative to the older reference, which fp32 / bf16 hold easily, and the
// row maximum is not computed at all.
#pragma once
#include <cuda.h>
#include "lg_common.cuh"
#include "lg_pattern.h"

namespace lg {

struct FwdArgs {
  const int32_t* tile_ent;   // kb * 16 + member mask (bit r: pattern row r of the super-tile has the block)
  const TileRec* order;      // [n_super_tiles] by launch rank
  __nv_bfloat16* o;
  float* lse;                // [B, Hq, L]
  unsigned int* error_word;  // first word of the workspace header
  unsigned long long expect_fp, expect_fp2;   // fingerprints of the lists this call was told the workspace holds (0: built by the call itself)
  int n_tiles, nB, n_list;   // sizes of the schedule arrays: tiles, pattern blocks, entries (bounds of the checked build)
  int64_t o_strides[3];      // batch, head, token (elements)
  int L, Hq, G;              // G = Hq / Hkv
  int q_start, Lq;           // queries exist for rows [q_start, q_start + Lq) of the L key positions only
                             // (a chunk served against a cache); Q, O, LSE are indexed by row - q_start
  int row_origin;            // first row of super-tile 0 (at most q_start)
  int exact_w, ns;           // token-exact window (0: off) and number of sink blocks
  int win_block, win_phase;  // with exact_w: the window edge is block-aligned in shifted coordinates instead --
                             // row i keeps the keys j with (i + phase) / win_block - (j + phase) / win_block
                             // < exact_w / win_block (a chunk served against a ring whose first kept token
                             // is `phase` tokens into the sequence); win_block = 0: token-exact edge
  const int32_t* doc_start;  // [B, L] first position of each query's document, or null
  float scale_log2;          // scale * log2(e)
  int head_group;            // heads whose CTAs run side by side (cta_coords); >= gridDim.x: all of them
  FwdSplit split;            // tiles cut along their keys
};

constexpr int kFwdTmaWarp = 8, kFwdMmaWarp0 = 9;
constexpr int kFwdThreads = 11 * 32;
constexpr float kFwdMaxProb = 256.0f;   // a half's probabilities may grow to this (relative to the row's reference) before the reference moves
constexpr int fwd_ctas_per_sm(int bufs) { return bufs == 1 ? 2 : 1; }   // one score buffer per slot: the form of which two share an SM
template <int D>
struct FwdSmem {
  static constexpr int kBox = 128 * 128;               // one 64-column box of 128 rows
  static constexpr int kTile = (D / 64) * kBox;        // 128 rows x D bf16
  static constexpr int kKStages = 3, kVStages = 2;
  static constexpr int oQ = 0;                         // [2 slots]
  static constexpr int oK = 2 * kTile;
  static constexpr int oV = oK + kKStages * kTile;
  static constexpr int oBar = oV + kVStages * kTile;
  static constexpr int kTotal = oBar + 256;
};

// Pieces of a tile that walks n_steps steps and is one of the ranks that are cut.
__device__ __forceinline__ int fwd_pieces(const FwdSplit& k, int n_steps) { return n_steps > k.len ? min((n_steps + k.len - 1) / k.len, k.places) : 1; }

// Joins the pieces of a cut tile inside its cluster.  Every CTA has laid its sums as they stand into its own shared memory, a row
// of D + 4 floats each (writes of a lane per row and reads along a row both without bank conflicts), and the rows'
// (reference, sum of probabilities) behind them; the CTA of piece `seg` adds its share of the 256 rows over all pieces, in
// their order, and writes O and LSE.  Nothing of it lies in global memory: calls that share a workspace share lists only.
template <int D>
struct FwdJoin {
  static constexpr int kRow = (D + 4) * 4, oMl = 256 * kRow, kBytes = oMl + 256 * 8;
};
// Rows r0, r0 + step, .. below `end` of a tile of up to N pieces, kBatch of them at a time: a load from another SM takes 1000
// cycles, so that one row after the other the share of a CTA took 6-8 us (4 heads x 3318 tokens, full causal, D = 128, two
// pieces a tile: 45.1 us, in batches 41.1).
template <int D, int N, int kBatch>
__device__ __forceinline__ void fwd_join_rows(const FwdArgs& a, uint32_t base, int n_segs, int b, int h, int row0, int r0, int end, int step, int c) {
  for (; r0 < end; r0 += kBatch * step) {
    float2 pair[kBatch][N];
    float4 v[kBatch][N];
#pragma unroll
    for (int x = 0; x < kBatch; ++x)
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const int r = r0 + x * step;
        pair[x][i] = make_float2(-INFINITY, 0.f);
        if (i < n_segs && r < end) {
          const uint32_t peer = cluster_addr(base, i);
          pair[x][i] = cluster_ld64(peer + FwdJoin<D>::oMl + r * 8);
          v[x][i] = cluster_ld128(peer + r * FwdJoin<D>::kRow + c * 16);
        }
      }
#pragma unroll
    for (int x = 0; x < kBatch; ++x) {
      float m = -INFINITY, l = 0.f;
#pragma unroll
      for (int i = 0; i < N; ++i) m = fmaxf(m, pair[x][i].x);
      const float mu = m == -INFINITY ? 0.f : m;
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const float w = fast_exp2(pair[x][i].x - mu);             // (0 for a piece no key of which the row sees,
        l += w * pair[x][i].y;
        if (pair[x][i].x == -INFINITY) continue;                  // which may not have written its sums)
        acc.x += w * v[x][i].x; acc.y += w * v[x][i].y; acc.z += w * v[x][i].z; acc.w += w * v[x][i].w;
      }
      const float inv = l > 0.f ? 1.f / l : l;                    // 0 where the row sees nothing, NaN stays NaN
      const int r = r0 + x * step, q = row0 + r;
      if (r < end && q < a.L && q >= a.q_start) {
        *reinterpret_cast<uint2*>(a.o + b * a.o_strides[0] + h * a.o_strides[1] + static_cast<int64_t>(q - a.q_start) * a.o_strides[2] + c * 4) =
            make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv));
        if (c == 0) a.lse[(static_cast<int64_t>(b) * a.Hq + h) * a.Lq + q - a.q_start] = l > 0.f ? (m + log2f(l)) * 0.6931471805599453f : -INFINITY;
      }
    }
  }
}
template <int D>
__device__ __forceinline__ void fwd_join(const FwdArgs& a, uint32_t base, uint32_t failed_flag, int seg, int n_segs, int b, int h, int row0) {
  constexpr int kLanes = D / 4, kRows = 32 / kLanes;              // lanes of a row (four columns each), rows of a warp
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = lane % kLanes;
  uint32_t failed = 0;
  for (int i = 0; i < n_segs; ++i) failed |= cluster_ld32(cluster_addr(failed_flag, i));
  if (failed) return;                                             // a piece was given up: the status word says so
  const int first = 256 * seg / n_segs + warp * kRows + lane / kLanes, end = 256 * (seg + 1) / n_segs, step = kFwdThreads / 32 * kRows;
  if (n_segs <= 2) fwd_join_rows<D, 2, 6>(a, base, n_segs, b, h, row0, first, end, step, c);
  else if (n_segs <= 4) fwd_join_rows<D, 4, 4>(a, base, n_segs, b, h, row0, first, end, step, c);
  else fwd_join_rows<D, 8, 2>(a, base, n_segs, b, h, row0, first, end, step, c);
}

template <int D, int BS, int NB /* score buffers per slot */, bool kSplit>
__global__ void __launch_bounds__(kFwdThreads, fwd_ctas_per_sm(NB))
fwd_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
           const __grid_constant__ CUtensorMap tm_v, const FwdArgs a) {
  using SM = FwdSmem<D>;
  constexpr int R4 = 256 / BS;                  // pattern rows per super-tile (2 or 4)
  constexpr int RS = R4 / 2;                    // pattern rows per slot
  constexpr uint32_t kSlotMask = (1u << RS) - 1u;
  constexpr int kTile = SM::kTile;
  constexpr uint32_t kColS = 0, kSlotS = 64 * NB, kColO = 2 * kSlotS, kTmemCols = NB == 1 ? 256 : 512;
  // SF / PF / OD are indexed [slot * 2 + buffer].  A parity wait is only meaningful while the barrier
  // is at most one phase behind the waiter; per half buffer that holds by construction (the S
  // product that re-fills a half is queued behind the P V product that read it), which is why
  // "O is complete" is tracked per half as well.
  enum { B_Q = 0, B_KF = 1, B_KE = 4, B_VF = 7, B_VE = 9, B_SF = 11, B_PF = 15, B_OD = 19, B_DRAIN = 23, B_COUNT = 25 };

  extern __shared__ __align__(1024) uint8_t smem[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + SM::oBar);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + B_COUNT);   // address, an earlier failure, a failure of this CTA's piece
  static_assert(B_COUNT * 8 + 12 <= 256, "barrier area too small");
  static_assert(fwd_ctas_per_sm(NB) * (SM::kTotal + 1024) <= 228 * 1024 && kColO + 2 * D <= kTmemCols, "does not fit an SM");
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // same value, known to be warp-uniform
  pdl_trigger();
  pdl_wait();
  if ((smem_u32(smem) & 1023u) != 0) {   // the swizzled tiles need 1024-byte alignment
    if (tid == 0) atomicCAS(a.error_word, 0u, (2u << 24) | 1u);
    return;
  }
  // has a wait already given up in this call?  (read now, so that it travels with the loads below)
  unsigned int abort_word = 0;
  if (tid == 0) abort_word = *reinterpret_cast<volatile unsigned int*>(a.error_word);
  int cta_x, cta_y;   // (batch, query head) and launch rank of this CTA's super-tile
  int seg = 0;        // which piece of the tile
  bool cut = false;   // one of the ranks that are cut
  if constexpr (kSplit) {
    // a cluster of `places` CTAs per cut tile, then the other tiles one by one (and what fills up their last cluster)
    cta_x = static_cast<int>(blockIdx.x);
    const int y = static_cast<int>(blockIdx.y), n_cut = a.split.n_cut;
    cut = y < n_cut * a.split.places;
    seg = cut ? y % a.split.places : 0;
    cta_y = cut ? y / a.split.places : y - n_cut * (a.split.places - 1);
    if (cta_y >= a.n_tiles) return;
  } else {
    cta_coords(blockIdx.y * gridDim.x + blockIdx.x, gridDim.x, gridDim.y, a.head_group, cta_x, cta_y);
  }
  const TileRec rec = load_rec(a.order + cta_y);
  if (!lists_match(a.error_word, a.expect_fp, a.expect_fp2, 1u)) return;
  uint8_t* sQ = smem + SM::oQ;
  uint8_t* sK = smem + SM::oK;
  uint8_t* sV = smem + SM::oV;

  const int tile = checked(rec.a, 0, a.n_tiles - 1, a.error_word, 100);
  const int b = cta_x / a.Hq, h = cta_x % a.Hq, hk = h / a.G;
  const int ent_off = checked(rec.off, 0, a.n_list, a.error_word, 101);
  int n_ent = checked(rec.cnt, 0, a.n_list - ent_off, a.error_word, 102);
  const int32_t* ent = a.tile_ent + ent_off;
  const int row0 = a.row_origin + tile * 256;
  int n_steps = (BS == 128) ? n_ent : (n_ent + 1) / 2;
  const int n_segs = kSplit && cut ? fwd_pieces(a.split, n_steps) : 1;
  if (kSplit && seg >= n_segs) return;                     // an empty place (uniform over the CTA; the cluster's barriers count who is left)
  const bool joint = kSplit && n_segs > 1;                 // the same in all CTAs of the cluster that are left
  if (joint) {
    const int first = n_steps * seg / n_segs, end = n_steps * (seg + 1) / n_segs;
    ent += (128 / BS) * first;
    n_ent = min(n_ent - (128 / BS) * first, (128 / BS) * (end - first));
    n_steps = end - first;
  }

  // entries of the two halves of step j (0: nobody's member, also past the end)
  auto load_ent = [&](int j, int& e0, int& e1) {
    if (j >= n_steps) { e0 = e1 = 0; return; }
    if (BS == 128) { e0 = e1 = ent[j]; return; }
    e0 = ent[2 * j];
    e1 = (2 * j + 1 < n_ent) ? ent[2 * j + 1] : 0;   // odd tail: no second block
  };

  if (tid == 0) {
    mbar_init(bars + B_Q, 1);
    for (int i = 0; i < 3; ++i) { mbar_init(bars + B_KF + i, 1); mbar_init(bars + B_KE + i, 2); }   // both issuers release
    for (int i = 0; i < 2; ++i) {
      mbar_init(bars + B_VF + i, 1); mbar_init(bars + B_VE + i, 2);
      mbar_init(bars + B_DRAIN + i, 1);
    }
    for (int i = 0; i < 4; ++i) { mbar_init(bars + B_SF + i, 1); mbar_init(bars + B_PF + i, 4); mbar_init(bars + B_OD + i, 1); }
    mbar_fence_init();
    tmem_slot[1] = tmem_slot[2] = abort_word;
  }
  if (warp == kFwdMmaWarp0) {
    tmem_alloc(tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  if (tmem_slot[1] != 0) {   // after a failed wait the rest of the grid does nothing: the call ends in seconds, not minutes
    if (!joint) {
      if (warp == kFwdMmaWarp0) tmem_dealloc(tmem, kTmemCols);
      return;
    }
    n_steps = n_ent = 0;                                   // (others of the cluster may be waiting for me)
  }

  // of a softmax thread's row:
  float m_ref = -INFINITY;   // reference maximum (scaled, log2 domain) the probabilities are relative to
  float l_run = 0.f;
  int p0 = 0, p1 = 0;        // P tiles published per score buffer (barrier phases)
  if (warp == kFwdTmaWarp) {
    // ------------------------------ TMA producer ------------------------------------------
    if (lane == 0) {
      tma_prefetch_desc(&tm_q); tma_prefetch_desc(&tm_k); tma_prefetch_desc(&tm_v);
      mbar_expect_tx(bars + B_Q, 2 * kTile);
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int x = 0; x < D / 64; ++x)
          // rows before q_start lie outside the tensor and arrive as zeros (their results are never stored)
          tma_load_4d(sQ + s * kTile + x * SM::kBox, &tm_q, bars + B_Q, x * 64, row0 + s * 128 - a.q_start, h, b);
      auto load_step = [&](uint8_t* dst, const CUtensorMap* tm, uint64_t* bar, int kb0, int kb1) {
#pragma unroll
        for (int x = 0; x < D / 64; ++x) {
          tma_load_4d(dst + x * SM::kBox, tm, bar, x * 64, kb0 * BS, hk, b);
          if (BS == 64) tma_load_4d(dst + x * SM::kBox + 64 * 128, tm, bar, x * 64, kb1 * BS, hk, b);
        }
      };
      bool ok = true;
      int nk = 0, nv = 0;   // loads started
      int e_next = n_steps > 0 ? ent[0] : 0, e_next1 = (BS == 64 && n_ent > 1) ? ent[1] : e_next;
      for (int j = 0; j < n_steps; ++j) {
        const int sk = j % 3, sv = j & 1;
        const int kb0 = e_next >> 4, kb1 = e_next1 >> 4;
        if (j + 1 < n_steps) {   // fetch the next step's entries now; they are needed one step later
          const int i0 = (BS == 128) ? j + 1 : 2 * j + 2;
          e_next = ent[i0];
          e_next1 = (BS == 64) ? ent[min(i0 + 1, n_ent - 1)] : e_next;
        }
        if (j >= 3) ok = mbar_wait(bars + B_KE + sk, ((j / 3) - 1) & 1, a.error_word, 2);
        if (!ok) break;
        mbar_expect_tx(bars + B_KF + sk, kTile);
        load_step(sK + sk * kTile, &tm_k, bars + B_KF + sk, kb0, kb1);
        nk = j + 1;
        if (j >= 2) ok = mbar_wait(bars + B_VE + sv, ((j / 2) - 1) & 1, a.error_word, 3);
        if (!ok) break;
        mbar_expect_tx(bars + B_VF + sv, kTile);
        load_step(sV + sv * kTile, &tm_v, bars + B_VF + sv, kb0, kb1);
        nv = j + 1;
      }
      if (kSplit && !ok) tmem_slot[2] = 1;
      // every copy this thread started has landed before the CTA may exit
      mbar_wait(bars + B_Q, 0, a.error_word, 4);
      for (int j = max(nk - 3, 0); j < nk; ++j) mbar_wait(bars + B_KF + j % 3, (j / 3) & 1, a.error_word, 5);
      for (int j = max(nv - 2, 0); j < nv; ++j) mbar_wait(bars + B_VF + (j & 1), (j / 2) & 1, a.error_word, 6);
    }
  } else if (warp == kFwdMmaWarp0 || warp == kFwdMmaWarp0 + 1) {
    // ------------------------------ MMA issuer of one slot --------------------------------
    // The whole warp runs the loop (addresses and descriptors stay warp-uniform values); one
    // elected lane issues.  Both issuers arrive once per step on the K / V "empty" barriers,
    // whether or not their slot used the step, and only after having seen the step's tile
    // arrive: an idle issuer can then never be a whole ring turn ahead of the other one.
    const int s = warp - kFwdMmaWarp0;
    const bool lead = elect_one();
    constexpr uint32_t idesc_s = make_idesc_bf16(128, 64, 0, 0);
    constexpr uint32_t idesc_o = make_idesc_bf16(128, D, 0, 1);
    constexpr uint32_t kHalfRows = (64 * 128) >> 4;   // 64 rows of a box, in 16-byte units
    const uint32_t hi = desc_hi(1024);
    const uint32_t q_lo = desc_lo(smem_u32(sQ), 16) + s * (kTile >> 4), k_lo = desc_lo(smem_u32(sK), 16);
    const uint32_t v_mn_lo = desc_lo(smem_u32(sV), SM::kBox);
    const uint32_t t_s = tmem + kColS + s * kSlotS, t_o = tmem + kColO + s * D;
    bool ok = mbar_wait(bars + B_Q, 0, a.error_word, 7);
    int n_pv = 0;                 // P V products issued (accumulate flag)
    int pf0 = 0, pf1 = 0;         // uses of the two half buffers whose P V product was issued (barrier phases)
    int ce0 = 0, ce1 = 0, ne0, ne1, nn0, nn1;
    load_ent(0, ne0, ne1);
    load_ent(1, nn0, nn1);
    bool k_seen = false;          // the K tile of the step whose S products are being issued has arrived
#pragma unroll 1
    for (int j = -1; j < n_steps; ++j) {   // step -1 only issues S products of step 0
      bool v_seen = false;
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int buf = NB == 2 ? hf : 0;
        if ((static_cast<uint32_t>(hf ? ce1 : ce0) >> (s * RS)) & kSlotMask) {           // P V of half hf of step j
          const int sv = j & 1;
          if (!v_seen) { ok = ok && mbar_wait(bars + B_VF + sv, (j / 2) & 1, a.error_word, 9); v_seen = true; }
          ok = ok && mbar_wait(bars + B_PF + s * 2 + buf, (buf ? pf1 : pf0) & 1, a.error_word, 10);
          if (ok) {
            tc_fence_after();
            const uint32_t b_lo = v_mn_lo + sv * (kTile >> 4) + hf * 4 * (2048 >> 4);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              if (lead) mma_ts2(t_o, t_s + buf * 64 + kk * 8, b_lo + kk * (2048 >> 4), hi, idesc_o, (n_pv > 0) || (kk > 0));
          }
          if (lead) mma_commit(bars + B_OD + s * 2 + buf);
          ++n_pv;
          if (buf) ++pf1; else ++pf0;
        }
        if (hf == 1 && j >= 0) {
          if (!v_seen) ok = ok && mbar_wait(bars + B_VF + (j & 1), (j / 2) & 1, a.error_word, 9);
          if (lead) mma_commit(bars + B_VE + (j & 1));
        }
        // the S product that takes the buffer next: the same half of step j + 1, or (one buffer) the next half
        const int jn = (NB == 2 || hf == 1) ? j + 1 : j, hn = NB == 2 ? hf : 1 - hf;
        const int ne = NB == 2 ? (hf ? ne1 : ne0) : (hf ? ne0 : ce1);
        if (hn == 0) k_seen = false;
        if ((static_cast<uint32_t>(ne) >> (s * RS)) & kSlotMask) {
          const int sk = jn % 3;
          if (!k_seen) { ok = ok && mbar_wait(bars + B_KF + sk, (jn / 3) & 1, a.error_word, 8); k_seen = true; }
          if (ok) {
            tc_fence_after();
            const uint32_t b_lo = k_lo + sk * (kTile >> 4) + hn * kHalfRows;
#pragma unroll
            for (int k = 0; k < D / 16; ++k) {
              constexpr int kB = SM::kBox >> 4;
              const uint32_t off = (k >> 2) * kB + (k & 3) * 2;
              if (lead) mma_ss2(t_s + buf * 64, q_lo + off, b_lo + off, hi, idesc_s, k > 0);
            }
          }
          if (lead) mma_commit(bars + B_SF + s * 2 + buf);
        }
        if (hn == 1 && jn >= 0 && jn < n_steps) {
          if (!k_seen) ok = ok && mbar_wait(bars + B_KF + jn % 3, (jn / 3) & 1, a.error_word, 8);
          if (lead) mma_commit(bars + B_KE + jn % 3);
        }
      }
      ce0 = ne0; ce1 = ne1;
      ne0 = nn0; ne1 = nn1;
      load_ent(j + 3, nn0, nn1);   // read ahead: off the critical path
    }
    if (kSplit && !ok) tmem_slot[2] = 1;
    if (lead) mma_commit(bars + B_DRAIN + s);
    mbar_wait(bars + B_DRAIN + s, 0, a.error_word, 11);   // nothing of ours is still running at exit
  } else {
    // ------------------------------ softmax warps -----------------------------------------
    const int s = warp >> 2;                                 // slot
    const int r = (warp & 3) * 32 + lane;                    // row in the slot == TMEM lane
    const int qi = row0 + s * 128 + r;
    const int member = s * RS + (BS == 128 ? 0 : (r >> 6));  // pattern row of the super-tile
    const uint32_t lane_addr = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    const uint32_t my_s = lane_addr + kColS + s * kSlotS, my_o = lane_addr + kColO + s * D;
    // lowest key position this row may see outside what the pattern already excludes: the start of its
    // document (0 without documents)
    const int dstart = (a.doc_start && qi < a.L && qi >= a.q_start) ? a.doc_start[static_cast<int64_t>(b) * a.L + qi] : 0;
    // oldest key position the window lets this row see (blocks outside the sink)
    const int win_lo = a.win_block > 0
                           ? ((qi + a.win_phase) / a.win_block - a.exact_w / a.win_block + 1) * a.win_block - a.win_phase
                           : qi - a.exact_w + 1;
    // every P V product issued so far has completed (at most one per buffer can still be running)
    auto wait_o = [&](uint32_t site) {
      bool w = true;
      if (p0 > 0) w = mbar_wait_warp(bars + B_OD + s * 2, (p0 - 1) & 1, a.error_word, site);
      if (w && p1 > 0) w = mbar_wait_warp(bars + B_OD + s * 2 + 1, (p1 - 1) & 1, a.error_word, site);
      return w;
    };
    bool ok = true;
    int ne0, ne1;
    load_ent(0, ne0, ne1);
#pragma unroll 1
    for (int j = 0; j < n_steps && ok; ++j) {
      const int e0 = ne0, e1 = ne1;
      load_ent(j + 1, ne0, ne1);
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int e = hf ? e1 : e0;
        if (((static_cast<uint32_t>(e) >> (s * RS)) & kSlotMask) == 0) continue;   // uniform over the slot
        // visible columns of this half: lo <= c < lim (the lower bound only exists with a
        // token-exact window, on blocks outside the sink)
        const int key0 = (e >> 4) * BS + (BS == 128 ? 64 * hf : 0);
        const int lim = ((e >> member) & 1) ? min(max(qi - key0 + 1, 0), 64) : 0;
        const int lo_abs = (a.exact_w > 0 && (e >> 4) >= a.ns) ? max(dstart, win_lo) : dstart;
        const int lo = min(max(lo_abs - key0, 0), 64);

        const bool masked = __any_sync(0xffffffffu, lim < 64 || lo > 0);   // (voted before the wait: off the chain)
        const int buf = NB == 2 ? hf : 0;
        ok = mbar_wait_warp(bars + B_SF + s * 2 + buf, (buf ? p1 : p0) & 1, a.error_word, 12);
        if (!ok) break;
        tc_fence_after();
        constexpr int C = 32 * NB;                   // columns in registers at a time
        uint32_t v[C];
        auto load_cols = [&](int c0) {               // columns c0 .. c0 + C - 1 of the half
#pragma unroll
          for (int x = 0; x < C; x += 32) tmem_ld32(my_s + buf * 64 + c0 + x, v + x);
          tmem_ld_wait();
          if (masked) {
#pragma unroll
            for (int y = 0; y < C; y += 32) {
              const uint32_t seen = bit_range(min(max(lo - c0 - y, 0), 32), min(max(lim - c0 - y, 0), 32));
#pragma unroll
              for (int x = 0; x < 32; ++x)
                v[y + x] = (seen >> x) & 1 ? v[y + x] : 0xff800000u;   // -inf: the exponential below gives exactly 0
            }
          }
        };
        // Probabilities relative to the reference as it stands; the row maximum is only looked at when
        // that cannot be right: the row has no reference yet, or the sum of the half's probabilities
        // (an upper bound of each of them) passes 2^8.  Otherwise every probability is below 2^8 and the
        // reference stays -- the maximum, its 32 instructions per row and the vote are off the common path.
        uint32_t preg[32];
        float psum;
        bool loaded = false;                         // with one chunk, v still holds the half when it is worked again
        auto exp_half = [&](float neg_m) {
          float q0 = 0.f, q1 = 0.f, q2 = 0.f, q3 = 0.f;   // independent partial sums
#pragma unroll
          for (int c0 = 0; c0 < 64; c0 += C) {
            if (NB == 1 || !loaded) { load_cols(c0); loaded = true; }
#pragma unroll
            for (int x = 0; x < C; x += 4) {
              const float x0 = fmaf(__uint_as_float(v[x]), a.scale_log2, neg_m);
              const float x1 = fmaf(__uint_as_float(v[x + 1]), a.scale_log2, neg_m);
              const float x2 = fmaf(__uint_as_float(v[x + 2]), a.scale_log2, neg_m);
              const float x3 = fmaf(__uint_as_float(v[x + 3]), a.scale_log2, neg_m);
              const float e0 = fast_exp2(x0), e1 = fast_exp2(x1), e2 = fast_exp2(x2), e3 = fast_exp2(x3);
              q0 += e0; q1 += e1; q2 += e2; q3 += e3;
              preg[(c0 + x) >> 1] = pack_bf16(e0, e1);
              preg[((c0 + x) >> 1) + 1] = pack_bf16(e2, e3);
            }
          }
          psum = (q0 + q2) + (q1 + q3);
        };
        const bool unset = (m_ref == -INFINITY);
        exp_half(unset ? 0.f : -m_ref);
        // (an unset reference with every column masked gives zeros and stays unset; NaN compares false
        // and cannot appear: masked scores are -inf, whose exponential is 0)
        const bool look = unset ? (lim > lo) : !(psum <= kFwdMaxProb);
        if (__any_sync(0xffffffffu, look)) {
          float mx = -INFINITY;
#pragma unroll
          for (int c0 = 0; c0 < 64; c0 += C) {
            if (NB == 1) load_cols(c0);
            float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll
            for (int x = 0; x < C; x += 8) {
              m0 = max3(m0, __uint_as_float(v[x + 0]), __uint_as_float(v[x + 1]));
              m1 = max3(m1, __uint_as_float(v[x + 2]), __uint_as_float(v[x + 3]));
              m2 = max3(m2, __uint_as_float(v[x + 4]), __uint_as_float(v[x + 5]));
              m3 = max3(m3, __uint_as_float(v[x + 6]), __uint_as_float(v[x + 7]));
            }
            mx = max3(mx, fmaxf(m0, m1), fmaxf(m2, m3));
          }
          // the rows that asked move their reference to the maximum seen so far (the others keep theirs)
          const float m_new = fmaxf(m_ref, mx * a.scale_log2);
          const bool raise = look && m_new > m_ref;
          const float alpha = raise ? fast_exp2(m_ref - m_new) : 1.f;   // m_ref = -inf -> 0
          if (raise) { m_ref = m_new; l_run *= alpha; }
          if (p0 + p1 > 0) {   // O already holds products: wait for them, then rescale my row
            ok = wait_o(13);
            if (!ok) break;
            tc_fence_after();
#pragma unroll 1
            for (int c = 0; c < D / 16; ++c) {
              uint32_t oreg[16];
              tmem_ld16(my_o + c * 16, oreg);
              tmem_ld_wait();
#pragma unroll
              for (int x = 0; x < 16; ++x) oreg[x] = __float_as_uint(__uint_as_float(oreg[x]) * alpha);
              tmem_st16(my_o + c * 16, oreg);
            }
          }
          exp_half((m_ref == -INFINITY) ? 0.f : -m_ref);
        }
        l_run += psum;
        tmem_st32(my_s + buf * 64, preg);   // P over the first columns of this half's S
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bars + B_PF + s * 2 + buf);
        if (buf) ++p1; else ++p0;
      }
    }
    // ---- epilogue: O / l -> bf16, LSE ------------------------------------------------------
    if (ok) ok = wait_o(14);
    if (joint) {                                             // a piece's sums stay as they are until both slots are done
      if (!ok) tmem_slot[2] = 1;
      ok = false;                                            // (the rows are not mine to write)
    }
    // warp-uniform condition (the tensor-memory loads below need the whole warp): some row of the warp
    // is a real query; rows past L or before q_start load with the others and store nothing
    if (ok && p0 + p1 > 0 && qi - lane < a.L && qi - lane + 32 > a.q_start) {
      const bool mine = qi < a.L && qi >= a.q_start;
      tc_fence_after();
      const float inv_l = l_run > 0.f ? 1.f / l_run : 0.f;
      // rows leave through the slot's own Q tile (its last S product is done: it precedes the last P V in
      // the issuer's queue), 4 KB per warp, so that the stores cover whole rows (store_acc_64cols)
      uint8_t* stage = sQ + s * kTile + (warp & 3) * 4096;
      const int q_first = row0 + s * 128 + (warp & 3) * 32;        // the warp's first row
      __nv_bfloat16* obase = a.o + b * a.o_strides[0] + h * a.o_strides[1];
#pragma unroll
      for (int c = 0; c < D / 64; ++c)
        store_acc_64cols(my_o + c * 64, stage, inv_l, [&](int r2) -> __nv_bfloat16* {
          const int q2 = q_first + r2;
          return (q2 < a.L && q2 >= a.q_start) ? obase + static_cast<int64_t>(q2 - a.q_start) * a.o_strides[2] + c * 64 : nullptr;
        });
      if (mine)
        a.lse[(static_cast<int64_t>(b) * a.Hq + h) * a.Lq + qi - a.q_start] =
            l_run > 0.f ? (m_ref + log2f(l_run)) * 0.6931471805599453f : -INFINITY;
    }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (kSplit) {
    if (joint) {
      // all copies have landed and all products are done: the operand buffers hold the sums from here on
      static_assert(FwdJoin<D>::kBytes <= SM::oBar, "the sums fit where the operands were");
      tc_fence_after();
      if (warp < kFwdTmaWarp) {
        const int row = warp * 32 + lane;                  // slot, row of the slot
        if (p0 + p1 > 0) {                                 // (uniform over the slot)
          const uint32_t my_o = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16) + kColO + (warp >> 2) * D;
#pragma unroll
          for (int c = 0; c < D; c += 32) {
            uint32_t reg[32];
            tmem_ld32(my_o + c, reg);
            tmem_ld_wait();
#pragma unroll
            for (int x = 0; x < 32; x += 4)
              *reinterpret_cast<uint4*>(smem + row * FwdJoin<D>::kRow + (c + x) * 4) = make_uint4(reg[x], reg[x + 1], reg[x + 2], reg[x + 3]);
          }
        }
        *reinterpret_cast<float2*>(smem + FwdJoin<D>::oMl + row * 8) = make_float2(l_run == 0.f ? -INFINITY : m_ref, l_run);
        tc_fence_before();
      }
      cluster_sync();                                      // (threads of CTAs that have left are not waited for)
      fwd_join<D>(a, smem_u32(smem), smem_u32(tmem_slot + 2), seg, n_segs, b, h, row0);
      cluster_sync();                                      // nobody leaves while its sums are being read
    }
  }
  if (warp == kFwdMmaWarp0) tmem_dealloc(tmem, kTmemCols);
}

}  // namespace lg
