// The static block pattern (paper Section 3.1) at block granularity, and the closed forms its schedules
// are laid out with.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace lg {

// SMs of a B200, for rules that size a grid.  Fixed and not asked of the device: workspace sizes follow from some of them
// and must come out the same without a GPU, and so must the bits of a result.
constexpr int kSms = 148;

struct PatternDev {
  int nB;       // ceil(L / block)
  int mode;     // 0 full causal, 1 sink+window, 2 strided+local
  int ns, nw;   // sink blocks, window blocks (own block included; one more when the window is token-exact)
  int stride, nl;
  // Optional pruning by packed documents (read by the schedule kernels; null on the host and for plain patterns):
  // doc_start[i] of the one sequence the lists are built for, and the block size in tokens.
  const int* doc_start;
  int block;
};

// Block (qb, kb) holds at least one allowed (query, key) pair.  Causality needs kb <= qb
// (the diagonal block always contains the pair i == j); the rest of the predicate only
// depends on the block indices (Section 3.1 patterns; documents: doc_first_block in lg_index.cuh).
__host__ __device__ __forceinline__ bool block_active(const PatternDev& p, int qb, int kb) {
  if (kb > qb) return false;
  if (p.mode == 0) return true;
  if (p.mode == 1) return kb < p.ns || qb - kb < p.nw;
  return qb - kb < p.nl || kb % p.stride == 0;
}

// ---- closed forms of the pattern WITHOUT documents --------------------------------------------
// A row's list is a sink run or a comb plus a run that ends at the diagonal; a column's list is one run that
// starts at the diagonal.  Row and column starts therefore need no counting pass: each schedule's place is
// computed where it is needed.  Documents only shorten the lists (a row loses its oldest blocks, a column its
// last rows), so the same places hold for them.  (The values are bounded by the pattern's block count, which
// fits an int; products on the way to them need 64 bits.)

// sum over x = 0 .. n-1 of min(x + 1, w)
__host__ __device__ __forceinline__ int64_t ramp_sum(int64_t n, int64_t w) {
  if (n <= 0 || w <= 0) return 0;
  return n <= w ? n * (n + 1) / 2 : w * (w + 1) / 2 + (n - w) * w;
}

// blocks in the rows before qb (0 <= qb <= nB)
__host__ __device__ __forceinline__ int row_start(const PatternDev& p, int qb) {
  const int64_t n = qb;
  if (p.mode == 0) return static_cast<int>(n * (n + 1) / 2);
  if (p.mode == 1) return static_cast<int>(ramp_sum(n, p.nw) + ramp_sum(n - p.nw, p.ns));
  const int64_t y = n > p.nl ? n - p.nl : 0, q = y / p.stride, rem = y % p.stride;   // comb blocks older than the local run
  return static_cast<int>(ramp_sum(n, p.nl) + p.stride * (q * (q + 1) / 2) + rem * (q + 1));
}

// query blocks in column c's list: rows c .. c + col_len - 1
__host__ __device__ __forceinline__ int col_len(const PatternDev& p, int c) {
  const int all = p.nB - c;
  if (p.mode == 0 || (p.mode == 1 && c < p.ns) || (p.mode == 2 && c % p.stride == 0)) return all;
  const int w = p.mode == 1 ? p.nw : p.nl;
  return w < all ? w : all;
}

// Comb columns that are longer than the local run: the first n_long_cols multiples of the stride.
__host__ __device__ __forceinline__ int n_long_cols(const PatternDev& p) {
  return (p.mode == 2 && p.stride > 1 && p.nB > p.nl) ? (p.nB - p.nl + p.stride - 1) / p.stride : 0;
}

// sum over x = a .. b-1 (a <= b <= nB) of min(w, nB - x)
__host__ __device__ __forceinline__ int64_t capped_sum(int64_t nB, int64_t w, int64_t a, int64_t b) {
  int64_t t = nB - w + 1;                            // from here on nB - x < w
  t = t < a ? a : (t > b ? b : t);
  return w * (t - a) + (b - t) * nB - (b * (b - 1) - t * (t - 1)) / 2;
}

// blocks in the first j columns of a strided pattern that are no long comb columns (in ascending order)
__host__ __device__ __forceinline__ int64_t short_cols_sum(const PatternDev& p, int64_t j) {
  const int64_t n_long = n_long_cols(p);
  const int64_t flat = p.nB > p.nl ? p.nB - p.nl + 1 - n_long : 0;   // of them have the full local run (or more columns: none)
  if (j <= flat) return j * p.nl;
  const int64_t c0 = flat + n_long;                  // first column of the tail, where lists shrink by one per column
  return flat * p.nl + capped_sum(p.nB, p.nl, c0, c0 + (j - flat));
}

// blocks in the columns before c (0 <= c <= nB)
__host__ __device__ __forceinline__ int col_start(const PatternDev& p, int c) {
  const int64_t n = c, nB = p.nB;
  if (p.mode == 0 || (p.mode == 2 && p.stride == 1)) return static_cast<int>(n * nB - n * (n - 1) / 2);
  if (p.mode == 1) {
    const int64_t s = n < p.ns ? n : p.ns;
    return static_cast<int>(s * nB - s * (s - 1) / 2 + capped_sum(nB, p.nw, s, n));
  }
  int64_t m = (n + p.stride - 1) / p.stride;         // long comb columns before c
  const int64_t n_long = n_long_cols(p);
  if (m > n_long) m = n_long;
  return static_cast<int>(m * nB - p.stride * (m * (m - 1) / 2) + short_cols_sum(p, n - m));
}

// position of block (qb, c) of the pattern in its column lists: the number of its kept dS tile
__host__ __device__ __forceinline__ int col_pos(const PatternDev& p, int qb, int c) { return col_start(p, c) + (qb - c); }

// ---- kv tiles of the dK/dV pass ------------------------------------------------------------
// A kv tile holds R pattern columns (R = 128 / block).  With R = 2 the two columns of a tile should be seen by
// the same query blocks: columns are taken in the order kv_col(0), kv_col(1), ... and neighbours in it share a
// tile.  Full causal and sink + window pair neighbouring columns, whose lists differ in a block at either end
// (in the order of their lengths, documents pair columns of unrelated documents, whose lists have nothing in
// common: 32 heads x 32K tokens in documents of 4000 on average, dK/dV pass 2.16 -> 2.0 ms, dQ pass 0.86 -> 0.72).  A comb column of the strided pattern is attended by every later query
// block and its neighbour by a handful, so there the long comb columns come first and share tiles among
// themselves.  kv_col(k) for 0 <= k < nB is a permutation of the columns.
__host__ __device__ __forceinline__ int kv_col(const PatternDev& p, int R, int k) {
  const int n_long = R == 2 ? n_long_cols(p) : 0;
  if (n_long == 0) return k;
  if (k < n_long) return k * p.stride;
  const int j = k - n_long, q = j / (p.stride - 1);
  return q < n_long ? q * p.stride + 1 + j % (p.stride - 1) : j + n_long;
}

// blocks in the columns kv_col(0) .. kv_col(k - 1): an upper bound of what the schedules of the tiles before
// the one that starts with kv_col(k) hold
__host__ __device__ __forceinline__ int kv_start(const PatternDev& p, int R, int k) {
  const int n_long = R == 2 ? n_long_cols(p) : 0;
  if (n_long == 0) return col_start(p, k);
  const int64_t m = k < n_long ? k : n_long;
  return static_cast<int>(m * p.nB - p.stride * (m * (m - 1) / 2) + short_cols_sum(p, k - m));
}

// Steps (128 keys) that the forward walks for the super-tile of n pattern rows from r0 on: the union of the rows' lists.
__host__ __device__ __forceinline__ int fwd_tile_steps(const PatternDev& p, int r0, int n) {
  const int end = r0 + n < p.nB ? r0 + n : p.nB;               // one past the youngest row's diagonal
  int blocks = end;
  if (p.mode != 0) {
    const int w = p.mode == 1 ? p.nw : p.nl;
    const int lo = r0 - w + 1 > 0 ? r0 - w + 1 : 0;            // oldest block of the oldest row's run
    blocks = end - lo + (p.mode == 1 ? (p.ns < lo ? p.ns : lo) : (lo + p.stride - 1) / p.stride);
  }
  return (blocks * p.block + 127) / 128;
}

// Super-tiles of the forward that are cut along their keys, a CTA per piece: the tiles of the first n_cut launch ranks (the
// longest) into ceil(steps / len) nearly equal pieces, at most `places`.  The CTAs of a tile are one cluster, which adds the pieces.
constexpr int kFwdMaxCutTiles = 4 * kSms, kFwdMaxPieces = 8, kFwdMaxPlaces = 1024;
struct FwdSplit {
  int len;                        // 0: no tile is cut
  int n_cut, places;
};

// CTAs, of clusters of 2 .. 8 with an SM for each CTA, that are taken to run at one time: a little less than the 148, 135, 132, 130, 132,
// 105 and 120 that the occupancy calculator gives for whole clusters; places that stay empty leave in 2 us and count for nothing.
// Above that the clusters wait for one another: 4 heads x 3318 tokens, D = 128, in 3 pieces (104 CTAs) 37 us, in 4 (128) 45 us.
constexpr int kFwdClusterCtas[kFwdMaxPieces + 1] = {0, 148, 144, 132, 120, 112, 96, 80, 80};

// Cut the longest super-tiles?  In units of steps (1.8 us): a CTA costs about 3 besides its own (launch, first loads, epilogue), and
// adding two pieces 3 at D = 64 and 4.5 at D = 128, more pieces 1.5 more.  An SM's share of the pass is (all + 3 per CTA) / SMs.  Where
// the longest tile alone takes longer (few heads, long rows) the number of pieces is the one with the smallest estimate:
// one round of CTAs ends with its longest; several, which only pairs of CTAs fill without gaps, with an SM's share and
// half a piece that sticks out.  Tiles are cut where that is less than 9 / 10 of the longest tile.  Over 54 problems x 7 numbers of
// pieces the choice takes 39.8 us on average, the best number for each 38.7, uncut 48.5.
// heads: query heads times batch of the whole problem, so that a step worked in groups of heads gives the same bits.
inline FwdSplit fwd_split(const PatternDev& p, int D, int st_row0, int n_tiles, int64_t heads) {
  FwdSplit k{};
  constexpr int kCta = 3, kMinLen = 3, kScale = 32;            // (estimates in 32nds)
  const int rows = 256 / p.block;
  if (heads * n_tiles > kFwdMaxCutTiles) return k;             // (an SM's share then holds several tiles)
  int64_t all = 0;
  int longest = 0;
  for (int t = 0; t < n_tiles; ++t) {
    const int n = fwd_tile_steps(p, st_row0 + rows * t, rows);
    all += n;
    if (n > longest) longest = n;
  }
  if (longest < 8 || (all + kCta * n_tiles) * heads >= static_cast<int64_t>(longest + kCta) * kSms) return k;
  int64_t best = static_cast<int64_t>(longest + kCta) * kScale * 9 / 10;
  for (int pieces = 2; pieces <= kFwdMaxPieces; ++pieces) {
    const int len = (longest + pieces - 1) / pieces;
    if (len < kMinLen) break;
    int64_t ctas = 0, n_cut = 0;
    for (int t = 0; t < n_tiles; ++t) {
      const int n = fwd_tile_steps(p, st_row0 + rows * t, rows), segs = (n + len - 1) / len;
      ctas += segs;
      n_cut += segs > 1;
    }
    if (heads * n_cut * pieces > kFwdMaxPlaces) continue;
    const int join = (pieces == 2 ? 3 : 6) * kScale / 2 + 3 * kScale * D / 128;
    int64_t then = join + (len + kCta) * kScale;
    if (ctas * heads > kFwdClusterCtas[pieces]) {
      if (pieces > 2) continue;
      then = join + (all + (kCta + 1) * ctas) * heads * kScale / kSms + (len + kCta) * kScale / 2;
    }
    if (then >= best) continue;
    best = then;
    k.len = len;
    k.n_cut = static_cast<int>(n_cut);
    k.places = pieces;
  }
  return k;
}

// Query blocks that see a kv tile, i.e. the union of its columns' runs.
__host__ __device__ __forceinline__ int kv_tile_len(const PatternDev& p, int R, int t) {
  const int a = kv_col(p, R, R * t), na = col_len(p, a);
  if (R == 1 || 2 * t + 1 >= p.nB) return na;
  const int b = kv_col(p, R, 2 * t + 1), nb = col_len(p, b);
  const int lo = a < b ? a : b, first_end = lo == a ? a + na : b + nb, second = lo == a ? b : a;
  const int end = (a + na > b + nb) ? a + na : b + nb;
  return second <= first_end ? end - lo : na + nb;
}

// The dK/dV pass gives a kv tile to one CTA, which walks it for every query head of the group.  Where that leaves the
// chip waiting for the longest tiles they are cut: a tile of n items (query block x query head) into
// ceil(n / len) nearly equal pieces, one CTA each, whose partial sums the CTA that finishes last adds in the order
// of the pieces.  The launch ranks 0, 1, ... (tiles longest first) fall into regions; a rank of region i has places
// for segs[i] pieces (a power of two; places beyond a tile's pieces stay empty).
constexpr int kKvMaxRegions = 6, kKvMaxSegs = 32, kKvMaxPlaces = 65535;   // places: a grid's limit in y
struct KvSplit {
  int len;                        // 0: no tile is cut
  int n_regions;
  int first_rank[kKvMaxRegions + 1], first_place[kKvMaxRegions + 1], segs[kKvMaxRegions];
  int n_ranks, n_places;          // of the regions that cut (segs > 1): ranks, and places of pieces
};


// Cut the longest kv tiles?  In units of half-steps (64 queries x 128 keys): a CTA costs about 8 of them besides its
// own (prologue, first loads, epilogue), so an even share of the pass is (all + 8 per CTA) / SMs.  Tiles are cut when
// the longest one alone exceeds 1.1 such shares, into pieces of half a share, at least 16 (shorter pieces cost more in
// overhead than they balance).  Measured, whole step: 3 x 16 / 4 heads x 6001 tokens, window 1024, D = 64: 604 -> 564
// us; 16 / 4 heads x 4096 tokens, full causal with documents: 369 -> 313 us.
// kv_total: kv heads (times batch) of the whole problem, so that a step worked in groups of heads gives the same bits.
// A call evaluates this once (resolve); it walks the tiles at most twice and allocates nothing (evaluated three times
// with a sorted copy of the lengths, a backward call over 2 heads x 128K tokens, window 4096, took 75 us of host time; 26).
inline KvSplit kv_split(const PatternDev& p, int n_ktiles, int G, int64_t nnz, int kv_total) {
  KvSplit k{};
  constexpr int kCta = 8, kMinLen = 16;
  const int R = 128 / p.block, per_item = p.block / 64;        // half-steps of an item
  const int64_t per_entry = static_cast<int64_t>(G) * per_item;
  // a bound first, without looking at the tiles: none is longer than twice the rows, and two columns share entries
  if (per_entry * p.nB * 2 * kSms <= nnz / R * per_entry * kv_total) return k;
  int64_t all = 0, longest = 0;
  for (int t = 0; t < n_ktiles; ++t) {
    const int len = kv_tile_len(p, R, t);
    all += len;
    if (len > longest) longest = len;
  }
  longest *= per_entry;
  const int64_t share = (all * per_entry + static_cast<int64_t>(kCta) * n_ktiles) * kv_total / kSms;
  if (10 * (longest + kCta) <= 11 * (share + kCta)) return k;
  int64_t piece = share / 2 > kMinLen ? share / 2 : kMinLen;   // half-steps
  if (piece * kKvMaxSegs < longest) piece = (longest + kKvMaxSegs - 1) / kKvMaxSegs;
  const int64_t items = (piece + per_item - 1) / per_item;
  if (items * per_item >= longest) return k;
  k.len = static_cast<int>(items);
  // a region per number of places, the longest tiles first as they are launched (documents only shorten tiles)
  int tiles[kKvMaxRegions] = {};                                // with up to 2^i pieces
  for (int t = 0; t < n_ktiles; ++t) {
    const int64_t n = (static_cast<int64_t>(kv_tile_len(p, R, t)) * G + items - 1) / items;
    int i = 0;
    while ((1 << i) < n) ++i;
    ++tiles[i];
  }
  int rank = 0, place = 0;
  for (int i = kKvMaxRegions - 1; i >= 0; --i) {
    if (tiles[i] == 0) continue;
    k.first_rank[k.n_regions] = rank;
    k.first_place[k.n_regions] = place;
    k.segs[k.n_regions++] = 1 << i;
    rank += tiles[i];
    place += tiles[i] << i;
    if (i > 0) { k.n_ranks = rank; k.n_places = place; }
  }
  k.first_rank[k.n_regions] = rank;
  k.first_place[k.n_regions] = place;
  if (place > kKvMaxPlaces) return KvSplit{};                   // (one kv head and more than 8.3 million tokens)
  return k;
}

}  // namespace lg
