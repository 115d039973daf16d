// C-ABI entry points: validation, workspace layout, block-index builder launches.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <atomic>
#include <mutex>

#include "lg_common.cuh"
#include "lg_host.h"
#include "lg_index.cuh"

namespace lg {

static std::atomic<long long> g_kernel_launches{0};
void note_launch() { g_kernel_launches.fetch_add(1, std::memory_order_relaxed); }

lg_status check_arch() {
  int dev = 0, major = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return LG_ERR_CUDA;
  if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) return LG_ERR_CUDA;
  return major == 10 ? LG_OK : LG_ERR_ARCH;
}

static bool strides_all_zero(const int64_t s[3]) { return s[0] == 0 && s[1] == 0 && s[2] == 0; }

static lg_status fix_strides(const int64_t in[3], int H, int L, int D, int64_t out[3]) {
  if (strides_all_zero(in)) {
    out[2] = D;
    out[1] = static_cast<int64_t>(L) * D;
    out[0] = static_cast<int64_t>(H) * L * D;
    return LG_OK;
  }
  for (int i = 0; i < 3; ++i) {
    if (in[i] <= 0 || in[i] % 8 != 0) return LG_ERR_INVALID_ARG;
    out[i] = in[i];
  }
  if (out[2] < D) return LG_ERR_INVALID_ARG;
  return LG_OK;
}

// Packed documents with several sequences: the block lists are shared by the sequences of a call, and documents prune
// them per sequence; with documents and B > 1 a call therefore runs sequence by sequence, each with its own lists in
// its own slice of the workspace (long packed samples fill the GPU one at a time).  The status
// word of the call stays the first word of the whole workspace.
static bool per_sequence(const Resolved& r) { return r.doc_start != nullptr && r.B > 1; }

lg_status resolve(const lg_attn_params* p, Resolved* r, bool want_bwd, int kv_total) {
  if (!p || !r) return LG_ERR_INVALID_ARG;
  if (p->B < 1 || p->Hq < 1 || p->Hkv < 1 || p->L < 1 || p->Hq % p->Hkv != 0) return LG_ERR_INVALID_ARG;
  if (p->block != 64 && p->block != 128) return LG_ERR_INVALID_ARG;
  if (p->L < 1) return LG_ERR_INVALID_ARG;   // L need not be a multiple of the block: the last block is then partial
  if (p->D != 64 && p->D != 128) return LG_ERR_UNSUPPORTED;
  if (!(p->scale >= 0.f) || isinf(p->scale)) return LG_ERR_INVALID_ARG;
  r->B = p->B; r->Hq = p->Hq; r->Hkv = p->Hkv; r->L = p->L; r->D = p->D; r->block = p->block;
  r->mode = p->mode; r->G = p->Hq / p->Hkv;
  r->pat.nB = (p->L + p->block - 1) / p->block;
  r->pat.mode = p->mode;
  r->pat.ns = r->pat.nw = r->pat.stride = r->pat.nl = 0;
  r->pat.doc_start = nullptr;
  r->pat.block = p->block;
  r->exact_w = 0;
  r->win_block = r->win_phase = 0;
  switch (p->mode) {
    case LG_MODE_FULL_CAUSAL:
      break;
    case LG_MODE_SINK_WINDOW:
      if (p->sink_tokens < 0 || p->sink_tokens % p->block != 0) return LG_ERR_INVALID_ARG;
      if (p->window_tokens < p->block || p->window_tokens % p->block != 0) return LG_ERR_INVALID_ARG;
      if (p->window_exact != 0 && p->window_exact != 1) return LG_ERR_INVALID_ARG;
      r->pat.ns = p->sink_tokens / p->block;
      // a token-exact window of W tokens reaches into one more block (partially)
      r->pat.nw = p->window_tokens / p->block + (p->window_exact ? 1 : 0);
      r->exact_w = p->window_exact ? p->window_tokens : 0;
      break;
    case LG_MODE_STRIDED_LOCAL:
      if (p->stride_blocks < 1 || p->local_blocks < 1) return LG_ERR_INVALID_ARG;
      r->pat.stride = p->stride_blocks;
      r->pat.nl = p->local_blocks;
      break;
    default:
      return LG_ERR_INVALID_ARG;
  }
  r->scale = p->scale > 0.f ? p->scale : 1.0f / sqrtf(static_cast<float>(p->D));
  lg_status s;
  if ((s = fix_strides(p->q_strides, p->Hq, p->L, p->D, r->qs)) != LG_OK) return s;
  if ((s = fix_strides(p->k_strides, p->Hkv, p->L, p->D, r->ks)) != LG_OK) return s;
  if ((s = fix_strides(p->v_strides, p->Hkv, p->L, p->D, r->vs)) != LG_OK) return s;
  if ((s = fix_strides(p->o_strides, p->Hq, p->L, p->D, r->os)) != LG_OK) return s;
  r->n_qtiles = (p->L + 127) / 128;
  r->n_ktiles = (p->L + 127) / 128;
  r->n_stiles = (p->L + 255) / 256;
  r->st_row0 = 0;
  r->q_start = 0;
  r->Lq = p->L;
  if (reinterpret_cast<uintptr_t>(p->doc_start) & 3) return LG_ERR_INVALID_ARG;
  r->doc_start = p->doc_start;
  r->error_word = nullptr;
  if (p->lists_prepared != 0 && p->lists_prepared != 1) return LG_ERR_INVALID_ARG;
  r->lists_prepared = p->lists_prepared;
  r->expect_fp = r->expect_fp2 = 0;
  // nnz from the per-row counts of each pattern
  int64_t nnz = 0;
  const PatternDev& pt = r->pat;
  for (int qb = 0; qb < pt.nB; ++qb) {
    if (pt.mode == 0) {
      nnz += qb + 1;
    } else if (pt.mode == 1) {
      const int win = qb + 1 < pt.nw ? qb + 1 : pt.nw;
      const int below = qb + 1 - win;           // blocks older than the window
      nnz += win + (pt.ns < below ? pt.ns : below);
    } else {
      const int loc = qb + 1 < pt.nl ? qb + 1 : pt.nl;
      const int below = qb + 1 - loc;
      nnz += loc + (below + pt.stride - 1) / pt.stride;
    }
  }
  r->nnz = nnz;
  r->kv_total = kv_total > 0 ? kv_total : p->B * p->Hkv;
  if (nnz > 0x3fffffff || pt.nB > (1 << 20)) return LG_ERR_UNSUPPORTED;
  // (documents in several sequences: the passes run once per sequence)
  const int kv_alone = per_sequence(*r) ? r->kv_total / r->B : r->kv_total;
  r->fsplit = fwd_split_of(*r, static_cast<int64_t>(kv_alone) * r->G);
  r->split = want_bwd ? kv_split(pt, r->n_ktiles, r->G, nnz, kv_alone) : KvSplit{};
  return LG_OK;
}

// Heads whose CTAs the forward and the backward passes run side by side (cta_coords): groups of four where
// the tiles of a head take about the same time -- sink + window, the window at most a quarter of the
// sequence --, two heads at a time for full causal attention, and all n_x heads together otherwise (combs
// need the longest-first order over all heads).
int head_group(const Resolved& r, int n_x) {
  const bool uniform = r.mode == LG_MODE_SINK_WINDOW && static_cast<long long>(r.pat.nw + r.pat.ns) * 4 <= r.pat.nB;
  if (r.mode == LG_MODE_FULL_CAUSAL) return kHeadGroupFull < n_x ? kHeadGroupFull : n_x;
  return uniform && n_x > kHeadGroup ? kHeadGroup : n_x;
}

// SMs of the current device (looked up once per device)
int sm_count() {
  static int cached[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
  if (cached[dev] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) return -1;
    cached[dev] = n;
  }
  return cached[dev];
}

// Two backward variants compute the same gradients (see BwdVariant).  The two passes run everywhere.
// Keeping dS trades workspace and HBM traffic (2 bytes per visible pair, written once and read once, on
// a memory system the attention kernels otherwise leave idle) for the two recomputed products of the dQ
// pass.  It is the default when the dS buffer (of one sequence, where documents make them run one by one) takes at most
// LG_KEEP_DS_MAX_GB gigabytes (the buffer holds every block of the pattern in full); without the variable
// the limit is 40 % of the current device's memory (77 GB of a B200's 192e9 bytes: 64 query heads of the
// strided pattern at 128K, 73 GB, still keep dS), 48 GB where no device can be asked.
// LG_BWD_VARIANT = two_pass | keep_ds overrides the choice (read at every call; it must not change between
// a size query, a prepare and the calls that use them).
static size_t ds_bytes_of(const Resolved& r, size_t heads) {   // 2 bytes per pair of every block of the pattern and query head, plus one tile of zeros at the end
  return heads * static_cast<size_t>(r.nnz) * r.block * r.block * 2 + 128 * 64 * 2;
}
size_t ds_buffer_bytes(const Resolved& r) { return ds_bytes_of(r, static_cast<size_t>(r.B) * r.Hq); }

// largest dS buffer the default choice accepts, in bytes
double keep_ds_limit() {
  if (const char* m = getenv("LG_KEEP_DS_MAX_GB")) return atof(m) * 1e9;
  static double cached[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return 48e9; }
  if (cached[dev] == 0.0) {
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess || total_b == 0) { cudaGetLastError(); return 48e9; }
    cached[dev] = 0.4 * static_cast<double>(total_b);
  }
  return cached[dev];
}

BwdVariant bwd_variant(const Resolved& r) {
  const char* env = getenv("LG_BWD_VARIANT");
  if (env && strcmp(env, "two_pass") == 0) return kBwdTwoPass;
  if (env && strcmp(env, "keep_ds") == 0) return kBwdKeepDs;
  // (the buffer of the whole problem: its groups of heads run the same variant, and their buffers exist side by side)
  return static_cast<double>(ds_bytes_of(r, static_cast<size_t>(r.kv_total) * r.G)) <= keep_ds_limit() ? kBwdKeepDs : kBwdTwoPass;
}

WsLayout ws_layout(const Resolved& r, bool want_bwd) {
  WsLayout w{};
  size_t off = sizeof(WsHeader);
  auto take = [&](size_t bytes) {
    size_t o = off;
    off = align_up(off + bytes, 256);
    return o;
  };
  const size_t nnz = static_cast<size_t>(r.nnz);
  w.sq_off = take(r.n_stiles * 4);
  w.sq_cnt = take(r.n_stiles * 4);
  w.sq_ent = take(nnz * 4);
  w.sq_order = take(r.n_stiles * sizeof(TileRec));
  if (want_bwd) {
    const bool keep = bwd_variant(r) == kBwdKeepDs;
    w.qt_off = take(static_cast<size_t>(r.n_qtiles) * 4);
    w.qt_cnt = take(static_cast<size_t>(r.n_qtiles) * 4);
    w.qt_ent = take(nnz * (keep ? kDqEntInts : 1) * 4);
    w.qt_order = take(static_cast<size_t>(r.n_qtiles) * sizeof(TileRec));
    w.kt_off = take(static_cast<size_t>(r.n_ktiles) * 4);
    w.kt_cnt = take(static_cast<size_t>(r.n_ktiles) * 4);
    w.kt_ent = take(nnz * 4);
    w.kt_order = take(static_cast<size_t>(r.n_ktiles) * sizeof(TileRec));
    w.kt_cols = take(static_cast<size_t>(r.n_ktiles) * 2 * 4);
    if (r.doc_start) w.doc_end = take(static_cast<size_t>(r.B) * r.L * 4);
    w.delta = take(static_cast<size_t>(r.B) * r.Hq * align_up(r.L, 128) * 8);   // rows padded to whole tiles   // two planes: -LSE * log2 e and -delta per query row
    if (keep) w.ds_buf = take(ds_buffer_bytes(r));
    const KvSplit& split = r.split;
    if (split.len > 0) {
      const size_t heads = static_cast<size_t>(r.B) * r.Hkv;
      w.kv_part = take(heads * split.n_places * 2 * 128 * r.D * 4);
      w.kv_ticket = take(heads * split.n_ranks * 4);
    }
  }
  w.total = off;
  return w;
}

lg_status launch_index_build(const Resolved& r, int32_t* row_ptr, int32_t* col_idx, int32_t* col_ptr,
                             int32_t* row_idx, cudaStream_t stream) {
  index_fill_kernel<<<r.pat.nB + 1, 64, 0, stream>>>(r.pat, row_ptr, col_idx, col_ptr, row_idx); note_launch();
  return cudaGetLastError() == cudaSuccess ? LG_OK : LG_ERR_CUDA;
}

// Which lists a workspace holds: FNV-1a over everything the lists and schedules depend on.
unsigned long long pattern_fingerprint(const Resolved& r, bool has_bwd) {
  unsigned long long h = 1469598103934665603ull;
  auto mix = [&](unsigned long long v) {
    for (int i = 0; i < 8; ++i) { h ^= (v >> (8 * i)) & 0xffu; h *= 1099511628211ull; }
  };
  mix(static_cast<unsigned long long>(r.L)); mix(r.block); mix(r.mode); mix(r.pat.ns); mix(r.pat.nw);
  mix(r.pat.stride); mix(r.pat.nl); mix(r.exact_w); mix(has_bwd ? 1 : 0);
  mix(reinterpret_cast<uintptr_t>(r.doc_start)); mix(r.doc_start ? r.B : 0);
  mix(has_bwd ? static_cast<int>(bwd_variant(r)) : 0);
  return h ? h : 1;
}

__global__ void header_begin_kernel(WsHeader* h) { header_begin(h); }

lg_status begin_workspace(uint8_t* ws, cudaStream_t stream) {
  header_begin_kernel<<<1, 1, 0, stream>>>(reinterpret_cast<WsHeader*>(ws)); note_launch();
  return cudaGetLastError() == cudaSuccess ? LG_OK : LG_ERR_CUDA;
}

lg_status prepare_workspace(const Resolved& r, const WsLayout& w, uint8_t* ws, int what, bool begin,
                            unsigned long long fp, cudaStream_t stream, const RingCopy* copy) {
  const bool want_fwd = (what & 1) != 0, want_bwd = (what & 2) != 0;
  auto i32 = [&](size_t off) { return reinterpret_cast<int32_t*>(ws + off); };
  auto recs = [&](size_t off) { return reinterpret_cast<TileRec*>(ws + off); };
  SchedArgs a{};
  a.p = r.pat;
  // The lists are shared by all sequences of the batch, so documents can only prune them when there
  // is one sequence (the usual case for long packed samples); otherwise they stay the pattern's own.
  if (r.doc_start && r.B == 1) a.p.doc_start = r.doc_start;
  WsHeader* header = reinterpret_cast<WsHeader*>(ws);
  a.header = begin ? header : nullptr;
  a.R = 128 / r.block;
  a.L = r.L;
  if (want_fwd) {   // the forward walks super-tiles of 256 rows; the backward passes have their own schedules
    a.n_stiles = r.n_stiles; a.st_row0 = r.st_row0;
    a.sq_off = i32(w.sq_off); a.sq_cnt = i32(w.sq_cnt); a.sq_ent = i32(w.sq_ent); a.sq_order = recs(w.sq_order);
  }
  if (want_bwd) {
    a.n_qtiles = r.n_qtiles; a.n_ktiles = r.n_ktiles;
    a.keep_ds = bwd_variant(r) == kBwdKeepDs;
    a.qt_off = i32(w.qt_off); a.qt_cnt = i32(w.qt_cnt); a.qt_ent = i32(w.qt_ent); a.qt_order = recs(w.qt_order);
    a.kt_off = i32(w.kt_off); a.kt_cnt = i32(w.kt_cnt); a.kt_ent = i32(w.kt_ent); a.kt_order = recs(w.kt_order);
    a.kt_cols = i32(w.kt_cols);
    if (r.doc_start) {
      a.doc_start = r.doc_start;
      a.doc_end = i32(w.doc_end);
      a.n_doc = static_cast<int64_t>(r.B) * r.L;
    }
  }
  constexpr int kWarps = kSchedThreads / 32;
  if (copy) a.copy = *copy;
  const int64_t tiles = static_cast<int64_t>(a.n_stiles) + a.n_qtiles + a.n_ktiles;
  const int64_t warps = tiles + (a.n_doc + 31) / 32 + (a.copy.n + 31) / 32;
  if (warps > 0x7fffffffll) return LG_ERR_UNSUPPORTED;
  if (launch_kernel(true, sched_build_kernel, dim3(static_cast<unsigned>((warps + kWarps - 1) / kWarps)), kSchedThreads, 0, stream, a) != cudaSuccess)
    return LG_ERR_CUDA;
  a.header = header;
  if (launch_kernel(true, sched_order_kernel, dim3(static_cast<unsigned>((tiles + kWarps - 1) / kWarps)), kSchedThreads, 0, stream, a, fp) != cudaSuccess)
    return LG_ERR_CUDA;
  return LG_OK;
}

// ---- tensor maps ---------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

lg_status make_tmap(CUtensorMap* out, const void* base, int B, int H, int L, int D, const int64_t strides[3],
                    int box_rows) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return LG_ERR_CUDA;
  cuuint64_t dims[4] = {static_cast<cuuint64_t>(D), static_cast<cuuint64_t>(L), static_cast<cuuint64_t>(H),
                        static_cast<cuuint64_t>(B)};
  cuuint64_t gstr[3] = {static_cast<cuuint64_t>(strides[2]) * 2, static_cast<cuuint64_t>(strides[1]) * 2,
                        static_cast<cuuint64_t>(strides[0]) * 2};
  cuuint32_t box[4] = {64, static_cast<cuuint32_t>(box_rows), 1, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult rc = fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, gstr, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return rc == CUDA_SUCCESS ? LG_OK : LG_ERR_CUDA;
}


// ---- chunk served against a sink + window ring ----------------------------------------------
struct ChunkPlan {
  lg_attn_params ap;     // exact-window sink + window attention over the kept tokens and the chunk
  Resolved r;
  WsLayout w;
  int kept;              // tokens the ring holds = first query row
  size_t lin_bytes;      // one of K_lin / V_lin
  size_t o_k, o_v, total;
};

static lg_status plan_chunk(const lg_decode_params* p, int32_t T, int64_t n_before, ChunkPlan* c) {
  if (!p) return LG_ERR_INVALID_ARG;
  if (p->B <= 0 || p->Hq <= 0 || p->Hkv <= 0 || p->Hq % p->Hkv != 0) return LG_ERR_INVALID_ARG;
  if (p->D != 64 && p->D != 128) return LG_ERR_UNSUPPORTED;
  if (p->sink_tokens < 0 || p->window_tokens < 64 || T <= 0 || n_before < 0) return LG_ERR_INVALID_ARG;
  // the pattern is made of 64-token blocks: sink and window must be multiples of 64; the chunk and
  // the fill level of the ring may be anything
  if (p->sink_tokens % 64 || p->window_tokens % 64) return LG_ERR_UNSUPPORTED;
  if (p->block_tokens < 0) return LG_ERR_INVALID_ARG;
  if (p->block_tokens > 0 && (p->window_tokens % p->block_tokens || p->sink_tokens % p->block_tokens))
    return LG_ERR_INVALID_ARG;
  const int64_t cap = static_cast<int64_t>(p->sink_tokens) + p->window_tokens;
  const int64_t kept = n_before < cap ? n_before : cap;
  if (kept + T > (1 << 24)) return LG_ERR_UNSUPPORTED;
  c->kept = static_cast<int>(kept);
  lg_attn_params& ap = c->ap;
  memset(&ap, 0, sizeof(ap));
  ap.B = p->B; ap.Hq = p->Hq; ap.Hkv = p->Hkv; ap.D = p->D;
  ap.L = c->kept + T;
  ap.block = 64;
  ap.mode = LG_MODE_SINK_WINDOW;
  ap.sink_tokens = p->sink_tokens;
  ap.window_tokens = p->window_tokens;
  ap.window_exact = 1;
  ap.scale = p->scale;
  // Q and O hold the chunk's T rows only
  ap.q_strides[0] = ap.o_strides[0] = static_cast<int64_t>(p->Hq) * T * p->D;
  ap.q_strides[1] = ap.o_strides[1] = static_cast<int64_t>(T) * p->D;
  ap.q_strides[2] = ap.o_strides[2] = p->D;
  lg_status s = resolve(&ap, &c->r);
  if (s != LG_OK) return s;
  c->r.q_start = c->kept;
  // super-tiles start at the chunk's first 64-token block: with tiles counted from the start of the virtual
  // sequence a chunk that fits k of them would straddle k + 1, and the grid would hold the empty ones before it
  c->r.st_row0 = c->kept / ap.block;
  c->r.n_stiles = (ap.L - c->r.st_row0 * ap.block + 255) / 256;
  c->r.Lq = T;
  // Block-aligned window: every non-sink row v of the virtual sequence (kept tokens, then the chunk) is the
  // token at position v + (n_before - kept), so the block-granular edge of the real positions is a
  // block-aligned edge in coordinates shifted by that amount.  The lists stay those of the token-exact
  // window, which contains it.
  c->r.win_block = p->block_tokens;
  c->r.win_phase = p->block_tokens > 0 ? static_cast<int>((n_before - kept) % p->block_tokens) : 0;
  c->r.fsplit = fwd_split_of(c->r, static_cast<int64_t>(p->B) * p->Hq);
  c->w = ws_layout(c->r, false);
  c->lin_bytes = align_up(static_cast<size_t>(p->B) * p->Hkv * ap.L * p->D * sizeof(__nv_bfloat16), 256);
  c->o_k = align_up(c->w.total, 256);
  c->o_v = c->o_k + c->lin_bytes;
  c->total = c->o_v + c->lin_bytes;
  return LG_OK;
}

// ---- self-test of the bounded wait -----------------------------------------------------------
// One thread waits on a barrier nobody will ever arrive at, with a limit of about a millisecond:
// the wait gives up, records its site in the error word and the kernel ends normally.
__global__ void wait_selftest_kernel(unsigned int* error_word, long long limit_cycles) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_fence_init();
    if (!mbar_try_wait(&bar, 0)) mbar_wait_slow(&bar, 0, error_word, 99, limit_cycles);
  }
}

static Resolved one_sequence(const Resolved& r, int b, void* workspace) {
  Resolved r1 = r;
  r1.B = 1;
  r1.kv_total = r.kv_total / r.B;
  r1.doc_start = r.doc_start + static_cast<int64_t>(b) * r.L;
  r1.error_word = r.error_word ? r.error_word : static_cast<unsigned int*>(workspace);
  return r1;
}

static size_t attn_workspace_total(const Resolved& r, bool want_bwd) {
  if (!per_sequence(r)) return ws_layout(r, want_bwd).total;
  return align_up(ws_layout(one_sequence(r, 0, nullptr), want_bwd).total, 256) * r.B;
}

size_t attn_workspace_bytes(const lg_attn_params* p, int want_bwd, int kv_total) {
  Resolved r;
  if (resolve(p, &r, want_bwd != 0, kv_total) != LG_OK) return 0;
  return attn_workspace_total(r, want_bwd != 0);
}

template <typename T>
static T* seq_ptr(T* base, int b, int64_t batch_stride_elems) {   // bf16 tensors: 2 bytes per element
  return base ? reinterpret_cast<T*>(reinterpret_cast<uint8_t*>(const_cast<void*>(static_cast<const void*>(base))) +
                                     static_cast<int64_t>(b) * batch_stride_elems * 2)
              : nullptr;
}
}  // namespace lg

using namespace lg;

extern "C" {

int64_t lg_block_index_nnz(const lg_attn_params* p) {
  Resolved r;
  lg_status s = resolve(p, &r);
  return s == LG_OK ? r.nnz : static_cast<int64_t>(s);
}

size_t lg_block_index_bytes(const lg_attn_params* p) {
  Resolved r;
  if (resolve(p, &r) != LG_OK) return 0;
  return (2 * (static_cast<size_t>(r.pat.nB) + 1) + 2 * static_cast<size_t>(r.nnz)) * sizeof(int32_t);
}

lg_status lg_build_block_index(const lg_attn_params* p, int32_t* row_ptr, int32_t* col_idx, int32_t* col_ptr,
                               int32_t* row_idx, int64_t* nnz_out_host, void* stream) {
  LG_RANGE("lg_build_block_index");
  Resolved r;
  lg_status s = resolve(p, &r);
  if (s != LG_OK) return s;
  if (!row_ptr || !col_idx || !col_ptr || !row_idx) return LG_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(row_ptr) | reinterpret_cast<uintptr_t>(col_idx) |
       reinterpret_cast<uintptr_t>(col_ptr) | reinterpret_cast<uintptr_t>(row_idx)) & 3)
    return LG_ERR_INVALID_ARG;
  if (nnz_out_host) *nnz_out_host = r.nnz;
  return launch_index_build(r, row_ptr, col_idx, col_ptr, row_idx, static_cast<cudaStream_t>(stream));
}

size_t lg_sparse_attn_workspace_bytes(const lg_attn_params* p, int want_bwd) { return attn_workspace_bytes(p, want_bwd, 0); }

int32_t lg_sparse_attn_bwd_variant(const lg_attn_params* p) {
  Resolved r;
  lg_status s = resolve(p, &r);
  if (s != LG_OK) return static_cast<int32_t>(s);
  return static_cast<int32_t>(bwd_variant(per_sequence(r) ? one_sequence(r, 0, nullptr) : r));
}

lg_status lg_sparse_attn_prepare(const lg_attn_params* p, void* workspace, size_t workspace_bytes, int want_bwd,
                                 void* stream) {
  LG_RANGE("lg_sparse_attn_prepare");
  Resolved r;
  lg_status s = resolve(p, &r, want_bwd != 0);
  if (s != LG_OK) return s;
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255)) return LG_ERR_INVALID_ARG;
  if (per_sequence(r)) return LG_ERR_UNSUPPORTED;   // lists per sequence: those calls build them themselves
  if (workspace_bytes < attn_workspace_total(r, want_bwd != 0)) return LG_ERR_WORKSPACE;
  if ((s = check_arch()) != LG_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  return prepare_workspace(r, ws_layout(r, want_bwd != 0), ws, want_bwd ? 3 : 1, true, pattern_fingerprint(r, want_bwd != 0), st);
}

}  // extern "C"

namespace lg {
lg_status attn_fwd_entry(const lg_attn_params* p, const void* q, const void* k, const void* v, void* o, float* lse,
                         void* workspace, size_t workspace_bytes, void* stream, unsigned int* status_word, int kv_total) {
  Resolved r;
  lg_status s = resolve(p, &r, false, kv_total);
  if (s != LG_OK) return s;
  r.error_word = status_word;
  if (!q || !k || !v || !o || !lse || !workspace) return LG_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o) || !aligned16(lse)) return LG_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(workspace) & 255) return LG_ERR_INVALID_ARG;
  if (workspace_bytes < attn_workspace_total(r, false)) return LG_ERR_WORKSPACE;
  if ((s = check_arch()) != LG_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  if (r.lists_prepared) {   // lists and schedules are in the workspace (the kernel checks the fingerprint)
    if (per_sequence(r)) return LG_ERR_UNSUPPORTED;
    r.expect_fp = pattern_fingerprint(r, false);
    r.expect_fp2 = pattern_fingerprint(r, true);
    return launch_fwd(r, ws_layout(r, false), q, k, v, o, lse, ws, st);
  }
  if (per_sequence(r)) {
    if ((s = begin_workspace(ws, st)) != LG_OK) return s;
    const size_t per = attn_workspace_total(r, false) / r.B;
    for (int b = 0; b < r.B; ++b) {
      const Resolved r1 = one_sequence(r, b, workspace);
      const WsLayout w1 = ws_layout(r1, false);
      uint8_t* wsb = ws + b * per;
      if ((s = prepare_workspace(r1, w1, wsb, 1, false, 0, st)) != LG_OK) return s;
      s = launch_fwd(r1, w1, seq_ptr(q, b, r.qs[0]), seq_ptr(k, b, r.ks[0]), seq_ptr(v, b, r.vs[0]),
                     seq_ptr(o, b, r.os[0]), lse + static_cast<int64_t>(b) * r.Hq * r.L, wsb, st);
      if (s != LG_OK) return s;
    }
    return LG_OK;
  }
  const WsLayout w = ws_layout(r, false);
  if ((s = prepare_workspace(r, w, ws, 1, true, 0, st)) != LG_OK) return s;
  return launch_fwd(r, w, q, k, v, o, lse, ws, st);
}

lg_status attn_bwd_entry(const lg_attn_params* p, const void* q, const void* k, const void* v, const void* o,
                         const float* lse, const void* d_o, void* dq, void* dk, void* dv, void* workspace,
                         size_t workspace_bytes, void* stream, cudaEvent_t* marks, unsigned int* status_word,
                         int kv_total) {
  Resolved r;
  lg_status s = resolve(p, &r, true, kv_total);
  if (s != LG_OK) return s;
  r.error_word = status_word;
  if (!q || !k || !v || !o || !lse || !d_o || !dq || !dk || !dv || !workspace) return LG_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o) || !aligned16(lse) || !aligned16(d_o) ||
      !aligned16(dq) || !aligned16(dk) || !aligned16(dv))
    return LG_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(workspace) & 255) return LG_ERR_INVALID_ARG;
  if (workspace_bytes < attn_workspace_total(r, true)) return LG_ERR_WORKSPACE;
  if ((s = check_arch()) != LG_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  if (r.lists_prepared) {
    if (per_sequence(r)) return LG_ERR_UNSUPPORTED;
    r.expect_fp = r.expect_fp2 = pattern_fingerprint(r, true);
    return launch_bwd(r, ws_layout(r, true), q, k, v, o, lse, d_o, dq, dk, dv, ws, st, marks);
  }
  if (per_sequence(r)) {
    if ((s = begin_workspace(ws, st)) != LG_OK) return s;
    const size_t per = attn_workspace_total(r, true) / r.B;
    for (int b = 0; b < r.B; ++b) {
      const Resolved r1 = one_sequence(r, b, workspace);
      const WsLayout w1 = ws_layout(r1, true);
      uint8_t* wsb = ws + b * per;
      if ((s = prepare_workspace(r1, w1, wsb, 2, false, 0, st)) != LG_OK) return s;
      s = launch_bwd(r1, w1, seq_ptr(q, b, r.qs[0]), seq_ptr(k, b, r.ks[0]), seq_ptr(v, b, r.vs[0]),
                     seq_ptr(o, b, r.os[0]), lse + static_cast<int64_t>(b) * r.Hq * r.L, seq_ptr(d_o, b, r.os[0]),
                     seq_ptr(dq, b, r.qs[0]), seq_ptr(dk, b, r.ks[0]), seq_ptr(dv, b, r.vs[0]), wsb, st,
                     b == 0 ? marks : nullptr);
      if (s != LG_OK) return s;
    }
    return LG_OK;
  }
  const WsLayout w = ws_layout(r, true);
  if ((s = prepare_workspace(r, w, ws, 2, true, 0, st)) != LG_OK) return s;
  return launch_bwd(r, w, q, k, v, o, lse, d_o, dq, dk, dv, ws, st, marks);
}

}  // namespace lg

extern "C" {

lg_status lg_sparse_attn_fwd(const lg_attn_params* p, const void* q, const void* k, const void* v, void* o,
                             float* lse, void* workspace, size_t workspace_bytes, void* stream) {
  LG_RANGE("lg_sparse_attn_fwd");
  return attn_fwd_entry(p, q, k, v, o, lse, workspace, workspace_bytes, stream, nullptr);
}

lg_status lg_sparse_attn_bwd(const lg_attn_params* p, const void* q, const void* k, const void* v, const void* o,
                             const float* lse, const void* d_o, void* dq, void* dk, void* dv, void* workspace,
                             size_t workspace_bytes, void* stream) {
  LG_RANGE("lg_sparse_attn_bwd");
  return attn_bwd_entry(p, q, k, v, o, lse, d_o, dq, dk, dv, workspace, workspace_bytes, stream, nullptr, nullptr);
}

lg_status lg_sparse_attn_bwd_marked(const lg_attn_params* p, const void* q, const void* k, const void* v,
                                    const void* o, const float* lse, const void* d_o, void* dq, void* dk, void* dv,
                                    void* workspace, size_t workspace_bytes, void* stream, void* const* events) {
  LG_RANGE("lg_sparse_attn_bwd_marked");
  if (!events) return LG_ERR_INVALID_ARG;
  cudaEvent_t ev[4];
  for (int i = 0; i < 4; ++i) {
    if (!events[i]) return LG_ERR_INVALID_ARG;
    ev[i] = static_cast<cudaEvent_t>(events[i]);
  }
  return attn_bwd_entry(p, q, k, v, o, lse, d_o, dq, dk, dv, workspace, workspace_bytes, stream, ev, nullptr);
}

size_t lg_chunk_prefill_workspace_bytes(const lg_decode_params* p, int32_t T, int64_t n_tokens_before) {
  ChunkPlan c;
  return plan_chunk(p, T, n_tokens_before, &c) == LG_OK ? c.total : 0;
}

lg_status lg_chunk_prefill(const lg_decode_params* p, const void* q_chunk, const void* k_chunk, const void* v_chunk,
                           const void* k_cache, const void* v_cache, int32_t T, int64_t n_tokens_before, void* o,
                           float* lse, void* workspace, size_t workspace_bytes, void* stream) {
  LG_RANGE("lg_chunk_prefill");
  ChunkPlan c;
  lg_status s = plan_chunk(p, T, n_tokens_before, &c);
  if (s != LG_OK) return s;
  if (!q_chunk || !k_chunk || !v_chunk || !o || !lse || !workspace) return LG_ERR_INVALID_ARG;
  if (c.kept > 0 && (!k_cache || !v_cache)) return LG_ERR_INVALID_ARG;
  if (!aligned16(q_chunk) || !aligned16(k_chunk) || !aligned16(v_chunk) || !aligned16(k_cache) ||
      !aligned16(v_cache) || !aligned16(o) || !aligned16(lse) || (reinterpret_cast<uintptr_t>(workspace) & 255))
    return LG_ERR_INVALID_ARG;
  if (workspace_bytes < c.total) return LG_ERR_WORKSPACE;
  if ((s = check_arch()) != LG_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  __nv_bfloat16* k_lin = reinterpret_cast<__nv_bfloat16*>(ws + c.o_k);
  __nv_bfloat16* v_lin = reinterpret_cast<__nv_bfloat16*>(ws + c.o_v);
  RingCopy copy;
  copy.k_cache = static_cast<const uint4*>(k_cache); copy.v_cache = static_cast<const uint4*>(v_cache);
  copy.k_chunk = static_cast<const uint4*>(k_chunk); copy.v_chunk = static_cast<const uint4*>(v_chunk);
  copy.k_lin = reinterpret_cast<uint4*>(k_lin); copy.v_lin = reinterpret_cast<uint4*>(v_lin);
  copy.n = static_cast<int64_t>(p->B) * p->Hkv * c.ap.L * (p->D / 8);
  copy.row_chunks = p->D / 8;
  copy.sink = p->sink_tokens; copy.window = p->window_tokens; copy.kept = c.kept; copy.T = T;
  copy.n_before = n_tokens_before;
  if ((s = prepare_workspace(c.r, c.w, ws, 1, true, 0, st, &copy)) != LG_OK) return s;
  return launch_fwd(c.r, c.w, q_chunk, k_lin, v_lin, o, lse, ws, st);
}

lg_status lg_selftest_wait_timeout(void* workspace, void* stream) {
  LG_RANGE("lg_selftest_wait_timeout");
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255)) return LG_ERR_INVALID_ARG;
  lg_status s = check_arch();
  if (s != LG_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (cudaMemsetAsync(workspace, 0, 2 * sizeof(unsigned int), st) != cudaSuccess) return LG_ERR_CUDA;   // the status words only
  wait_selftest_kernel<<<1, 32, 0, st>>>(static_cast<unsigned int*>(workspace), 2000000ll); note_launch();
  return cudaGetLastError() == cudaSuccess ? LG_OK : LG_ERR_CUDA;
}

lg_status lg_last_status(void* workspace, void* stream) {
  LG_RANGE("lg_last_status");
  if (!workspace) return LG_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (cudaStreamSynchronize(st) != cudaSuccess) return LG_ERR_CUDA;
  unsigned int word[2] = {0, 0};   // error word of the latest call, and one an earlier call left unread
  if (cudaMemcpy(word, workspace, sizeof(word), cudaMemcpyDeviceToHost) != cudaSuccess) return LG_ERR_CUDA;
  if (word[0] != 0 || word[1] != 0) {
    if (cudaMemset(workspace, 0, sizeof(word)) != cudaSuccess) return LG_ERR_CUDA;
    const unsigned int first = word[1] != 0 ? word[1] : word[0];
    // 3: lists of another pattern; 4 (checked builds): a schedule value out of range -- either way the workspace is not
    // what the call needs
    return ((first >> 24) == 3u || (first >> 24) == 4u) ? LG_ERR_WORKSPACE : LG_ERR_DEVICE_TIMEOUT;
  }
  return LG_OK;
}

int64_t lg_debug_kernel_launches(void) { return g_kernel_launches.load(std::memory_order_relaxed); }

const char* lg_status_string(lg_status s) {
  switch (s) {
    case LG_OK: return "ok";
    case LG_ERR_INVALID_ARG: return "invalid argument";
    case LG_ERR_UNSUPPORTED: return "unsupported problem";
    case LG_ERR_WORKSPACE: return "workspace too small";
    case LG_ERR_CUDA: return "CUDA call failed";
    case LG_ERR_DEVICE_TIMEOUT: return "a bounded device-side wait expired";
    case LG_ERR_ARCH: return "device is not sm_100";
  }
  return "unknown status";
}

}  // extern "C"
