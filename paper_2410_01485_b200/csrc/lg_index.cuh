// Block-index builder: CSR / CSC lists of active blocks of the static pattern (paper
// Section 3.2: the mask lives in compressed-sparse-row form and is the same for all heads),
// and the per-tile schedules the attention kernels walk.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "lg_common.cuh"
#include "lg_pattern.h"

namespace lg {

// ---- CSR / CSC lists (lg_build_block_index) ---------------------------------------------------
// grid = nB + 1 blocks of 64 threads: block b writes row_ptr[b], col_ptr[b] (closed forms), and below nB warp 0
// writes row b (ascending kb) and warp 1 column b (ascending qb), by ordered ballot compaction.
__global__ void index_fill_kernel(PatternDev p, int32_t* __restrict__ row_ptr, int32_t* __restrict__ col_idx,
                                  int32_t* __restrict__ col_ptr, int32_t* __restrict__ row_idx) {
  const int b = blockIdx.x;
  const int lane = threadIdx.x & 31;
  const bool is_row = (threadIdx.x >> 5) == 0;
  const int start = is_row ? row_start(p, b) : col_start(p, b);
  if (lane == 0) (is_row ? row_ptr : col_ptr)[b] = start;
  if (b == p.nB) return;
  int32_t* out = (is_row ? col_idx : row_idx) + start;
  int written = 0;
  for (int base = 0; base < p.nB; base += 32) {
    const int x = base + lane;
    const bool on = x < p.nB && (is_row ? block_active(p, b, x) : block_active(p, x, b));
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (on) out[written + __popc(m & ((1u << lane) - 1))] = x;
    written += __popc(m);
  }
}

// ---- schedules -------------------------------------------------------------------------------
// Everything the attention kernels walk, in two launches: sched_build_kernel writes the entries of every tile (one
// warp per tile, straight from the block predicate -- the places come from the closed forms of lg_pattern.h, so
// nothing has to be counted or scanned first), sched_order_kernel ranks the tiles longest first.
//   super-tile (forward, 256 query rows = up to 4 pattern rows): ascending kv blocks, kb * 16 + member mask
//   query tile (dQ pass that recomputes, 128 rows):              ascending kv blocks, kb * 4 + member mask
//   kv tile (dK/dV pass, R pattern columns):                     ascending query blocks, qb * 4 + member mask
//   query tile (dQ pass that reads the kept dS):                 ascending kv tiles, see dq_entries below
// (member bit r: pattern row / column r of the tile has the block).

// A chunk served against a sink + window ring: time-ordered copy of what the ring holds, followed by the chunk,
// K_lin, V_lin [B, Hkv, kept + T, D].  Row v < kept is the cache slot of position
//   v                                   (v < sink: the sink never moves)
//   n_before - (kept - sink) + v - sink (the kept window tokens, oldest first),
// row v >= kept is chunk token v - kept.
struct RingCopy {
  const uint4 *k_cache, *v_cache, *k_chunk, *v_chunk;
  uint4 *k_lin, *v_lin;
  int64_t n;                 // 16-byte chunks of K_lin (0: no copy)
  int row_chunks;            // of a row: D / 8
  int sink, window, kept, T;
  int64_t n_before;
};

struct SchedArgs {
  PatternDev p;
  WsHeader* header;          // reset first (null: done by the caller)
  int R;                     // pattern rows / columns per 128 tokens
  int n_stiles, st_row0;     // super-tiles, and the pattern row the first one starts at
  int n_qtiles, n_ktiles;    // 0: no schedule of that kind
  int keep_ds;               // query tiles: the schedule over the kept dS instead of the recomputing pass's
  int32_t *sq_off, *sq_cnt, *sq_ent;
  int32_t *qt_off, *qt_cnt, *qt_ent;
  int32_t *kt_off, *kt_cnt, *kt_ent, *kt_cols;
  TileRec *sq_order, *qt_order, *kt_order;
  const int32_t* doc_start;  // with documents and a backward: doc_end[i] is derived for n_doc tokens, L per sequence
  int32_t* doc_end;
  int64_t n_doc;
  int L;
  RingCopy copy;
};

// Start of a call that (re)builds the lists: a header that was never initialised is reset, an
// error word nobody has read yet moves to `latched`, and the fingerprint is withdrawn until the
// lists are whole again.
__device__ __forceinline__ void header_begin(WsHeader* h) {
  // (memory that was a workspace before may hold the magic between words that were written over since)
  if (h->magic != kWsMagic || !is_status(h->latched)) { h->magic = kWsMagic; h->latched = 0; }
  else if (h->latched == 0 && is_status(h->error_word)) h->latched = h->error_word;
  h->error_word = 0;
  h->fingerprint = 0;
}

// Oldest block the documents leave to query block qb.  The first row of a query block belongs to the earliest document
// of the block, so it sees the most: a key block that ends before that document starts holds nothing any row of the
// block may see.  (A superset of the blocks that are really needed; what is left over is masked in the kernels.)
__device__ __forceinline__ int doc_first_block(const PatternDev& p, int qb) {
  return p.doc_start ? max(p.doc_start[qb * p.block], 0) / p.block : 0;
}

// The ascending union of the lists of pattern rows r0 .. r0 + n - 1 (n <= 4) as `kb * mul + member mask`; one warp.
__device__ __forceinline__ int merge_rows(const PatternDev& p, int r0, int n, int mul, int32_t* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  int first[4], lo = 0x7fffffff;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    first[r] = (r < n && r0 + r < p.nB) ? doc_first_block(p, r0 + r) : 0x7fffffff;
    lo = min(lo, first[r]);
  }
  const int hi = min(r0 + n, p.nB);                     // the youngest row's diagonal
  const int win0 = p.mode == 1 ? r0 - p.nw + 1 : 0;     // sink + window: nothing between the sink and the oldest row's window
  int written = 0;
  for (int base = lo & ~31; base < hi; base += 32) {
    if (p.mode == 1 && base >= p.ns && base + 32 <= win0) base = win0 & ~31;
    const int kb = base + lane;
    int mask = 0;
    if (kb < hi) {
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (kb >= first[r] && block_active(p, r0 + r, kb)) mask |= 1 << r;   // (first[r] = INT_MAX: no such row)
    }
    const unsigned m = __ballot_sync(0xffffffffu, mask != 0);
    if (mask) out[written + __popc(m & ((1u << lane) - 1))] = kb * mul + mask;
    written += __popc(m);
  }
  return written;
}

// Entries of query tile t for the dQ pass that reads the kept dS tiles.  The dK/dV pass leaves one dS tile per
// block of the pattern and 64-row half of its query block, numbered by the block's position p in the column
// lists (col_pos): 128-token blocks: tiles 2 p and 2 p + 1 (128 keys x 64 queries each); 64-token blocks: tile p
// (64 keys x 64 queries).  A query tile of 128 rows needs, for every kv tile T with an active column in the row(s)
// of its query block(s), the four quarters (64-row half m, 64-key half n) of its 128 x 128 product; entry =
// (T, tile of (m, n) at 1 + 2 n + m), -1 where the pattern has no block (that quarter of dS is zero).  With
// 128-token blocks only n = 0 is used: the tiles of the two halves.  One warp, kv tiles ascending.
__device__ __forceinline__ int dq_entries(const PatternDev& p, int R, int n_ktiles, int t, int32_t* __restrict__ out) {
  constexpr int E = kDqEntInts;
  const int lane = threadIdx.x & 31;
  int first[2];
#pragma unroll
  for (int m = 0; m < 2; ++m) first[m] = (m < R && R * t + m < p.nB) ? doc_first_block(p, R * t + m) : 0x7fffffff;
  const bool in_order = R == 1 || n_long_cols(p) == 0;   // tile T holds columns R T, R T + 1
  const int lo = in_order ? min(first[0], first[1]) / R : 0, hi = in_order ? min(t + 1, n_ktiles) : n_ktiles;
  int written = 0;
  for (int base = lo & ~31; base < hi; base += 32) {
    const int T = base + lane;
    int q[4] = {-1, -1, -1, -1};
    bool any = false;
    if (T < hi) {
#pragma unroll
      for (int n = 0; n < 2; ++n) {
        if (n >= R || R * T + n >= p.nB) continue;
        const int c = kv_col(p, R, R * T + n);
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          const int qb = R * t + m;
          if (m >= R || c < first[m] || !block_active(p, qb, c)) continue;   // (first[m] = INT_MAX: no such row)
          q[2 * n + m] = col_pos(p, qb, c);
          any = true;
        }
      }
      if (R == 1 && any) { q[1] = 2 * q[0] + 1; q[0] = 2 * q[0]; }
    }
    const unsigned m = __ballot_sync(0xffffffffu, any);
    if (any) {
      int32_t* e = out + E * (written + __popc(m & ((1u << lane) - 1)));
      e[0] = T;
#pragma unroll
      for (int i = 0; i < 4; ++i) e[1 + i] = q[i];
    }
    written += __popc(m);
  }
  return written;
}

// The ascending union of the lists of a kv tile's columns as `qb * 4 + member mask`; one warp.
__device__ __forceinline__ int merge_cols(const PatternDev& p, int ca, int cb, int32_t* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int lo = cb >= 0 ? min(ca, cb) : ca;
  int hi = ca + col_len(p, ca);
  if (cb >= 0) hi = max(hi, cb + col_len(p, cb));
  int written = 0;
  for (int base = lo & ~31; base < hi; base += 32) {
    const int qb = base + lane;
    int mask = 0;
    if (qb < hi) {
      const int first = doc_first_block(p, qb);
      if (ca >= first && block_active(p, qb, ca)) mask |= 1;
      if (cb >= first && cb >= 0 && block_active(p, qb, cb)) mask |= 2;
    }
    const unsigned m = __ballot_sync(0xffffffffu, mask != 0);
    if (mask) out[written + __popc(m & ((1u << lane) - 1))] = qb * 4 + mask;
    written += __popc(m);
  }
  return written;
}

// end (one past the last token) of the document token j belongs to, from doc_start[i] = first token of token i's
// document (non-decreasing): the first i > j whose document starts after j, found by bisection, or L.
__device__ __forceinline__ int doc_end_of(const int32_t* ds, int j, int L) {
  int lo = j, hi = L;            // ds[lo] <= j (its own document); ds[hi] > j, with ds[L] taken as +inf
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (ds[mid] > j) hi = mid; else lo = mid;
  }
  return hi;
}

// one 16-byte chunk of K and of V
__device__ __forceinline__ void ring_linearise(const RingCopy& r, int64_t i) {
  const int Lc = r.kept + r.T;
  const int c = static_cast<int>(i % r.row_chunks), v = static_cast<int>((i / r.row_chunks) % Lc);
  const int64_t bh = i / (static_cast<int64_t>(r.row_chunks) * Lc);
  if (v < r.kept) {
    const int64_t pos = v < r.sink ? v : r.n_before - (r.kept - r.sink) + (v - r.sink);
    const int64_t slot = pos < r.sink ? pos : r.sink + (pos - r.sink) % r.window;
    const int64_t off = (bh * (r.sink + r.window) + slot) * r.row_chunks + c;
    r.k_lin[i] = r.k_cache[off];
    r.v_lin[i] = r.v_cache[off];
  } else {
    const int64_t off = (bh * r.T + (v - r.kept)) * r.row_chunks + c;
    r.k_lin[i] = r.k_chunk[off];
    r.v_lin[i] = r.v_chunk[off];
  }
}

constexpr int kSchedThreads = 256;   // warps are independent of one another

// Latency-bound integer work: a warp per tile looks at 32 blocks at a time (the one-thread-per-tile merges this
// replaces took 30 us of a 520 us chunk call and 260 us of a 4.8 ms step over packed documents).
__global__ void __launch_bounds__(kSchedThreads) sched_build_kernel(const SchedArgs a) {
  pdl_trigger();
  pdl_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0 && a.header) header_begin(a.header);
  const int lane = threadIdx.x & 31;
  int64_t w = static_cast<int64_t>(blockIdx.x) * (kSchedThreads / 32) + (threadIdx.x >> 5);
  if (w < a.n_stiles) {
    const int t = static_cast<int>(w), r0 = a.st_row0 + 2 * a.R * t;
    const int off = row_start(a.p, r0) - row_start(a.p, a.st_row0);
    const int n = merge_rows(a.p, r0, 2 * a.R, 16, a.sq_ent + off);
    if (lane == 0) { a.sq_off[t] = off; a.sq_cnt[t] = n; }
    return;
  }
  w -= a.n_stiles;
  if (w < a.n_qtiles) {
    const int t = static_cast<int>(w), off = row_start(a.p, a.R * t);
    const int n = a.keep_ds ? dq_entries(a.p, a.R, a.n_ktiles, t, a.qt_ent + static_cast<int64_t>(kDqEntInts) * off)
                            : merge_rows(a.p, a.R * t, a.R, 4, a.qt_ent + off);
    if (lane == 0) { a.qt_off[t] = off; a.qt_cnt[t] = n; }
    return;
  }
  w -= a.n_qtiles;
  if (w < a.n_ktiles) {
    const int t = static_cast<int>(w), k = a.R * t, off = kv_start(a.p, a.R, k);
    const int ca = kv_col(a.p, a.R, k), cb = (a.R == 2 && k + 1 < a.p.nB) ? kv_col(a.p, a.R, k + 1) : -1;   // -1: no second column
    const int n = merge_cols(a.p, ca, cb, a.kt_ent + off);
    if (lane == 0) {
      a.kt_off[t] = off; a.kt_cnt[t] = n;
      a.kt_cols[a.R * t] = ca;
      if (a.R == 2) a.kt_cols[2 * t + 1] = cb;
    }
    return;
  }
  w -= a.n_ktiles;
  int64_t i = w * 32 + lane;
  if (i < a.n_doc) {
    const int j = static_cast<int>(i % a.L);
    a.doc_end[i] = doc_end_of(a.doc_start + (i - j), j, a.L);
    return;
  }
  i -= (a.n_doc + 31) / 32 * 32;
  if (i >= 0 && i < a.copy.n) ring_linearise(a.copy, i);   // (a few schedule warps beside a copy: one launch for both)
}

// rank of tile t by (count descending, tile ascending); one warp
__device__ __forceinline__ int rank_of(const int32_t* cnt, int n, int t) {
  const int c = cnt[t];
  int rank = 0;
  for (int u = threadIdx.x & 31; u < n; u += 32) {
    const int cu = cnt[u];
    rank += (cu > c || (cu == c && u < t)) ? 1 : 0;
  }
  return __reduce_add_sync(0xffffffffu, rank);
}

// Launch order: tiles with more work first (order[rank] = what a CTA needs to know of the tile).  The last launch of a build: the header gets the
// fingerprint the lists are known by (0: none).
__global__ void __launch_bounds__(kSchedThreads) sched_order_kernel(const SchedArgs a, unsigned long long fp) {
  pdl_trigger();
  pdl_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0 && fp != 0) a.header->fingerprint = fp;
  int w = blockIdx.x * (kSchedThreads / 32) + (threadIdx.x >> 5);
  const int32_t* cnt[3] = {a.sq_cnt, a.qt_cnt, a.kt_cnt};
  const int32_t* off[3] = {a.sq_off, a.qt_off, a.kt_off};
  TileRec* order[3] = {a.sq_order, a.qt_order, a.kt_order};
  const int n[3] = {a.n_stiles, a.n_qtiles, a.n_ktiles};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (w < n[i]) {
      const int rank = rank_of(cnt[i], n[i], w);
      if ((threadIdx.x & 31) == 0) {
        TileRec r{off[i][w], cnt[i][w], w, -1};
        if (i == 2) { r.a = a.kt_cols[a.R * w]; r.b = a.R == 2 ? a.kt_cols[2 * w + 1] : -1; }
        order[i][rank] = r;
      }
      return;
    }
    w -= n[i];
  }
}

}  // namespace lg
