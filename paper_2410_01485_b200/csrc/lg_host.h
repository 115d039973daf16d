// Host-side helpers shared by the C-ABI entry points: validation, workspace layout,
// tensor-map encoding.  Nothing here is exported.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <atomic>

#include "../../include/lg.h"
#include "lg_pattern.h"

// Optional NVTX ranges around every entry point (build with -DLG_NVTX; the NVTX headers are
// self-contained and cost nothing when no tool is attached).
#ifdef LG_NVTX
#include <nvtx3/nvToolsExt.h>
namespace lg {
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
};
}  // namespace lg
#define LG_RANGE(name) ::lg::NvtxRange lg_nvtx_range_(name)
#else
#define LG_RANGE(name) ((void)0)
#endif

namespace lg {

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Diagnostic only: how many kernels the library has launched in this process (read through
// lg_debug_kernel_launches); nothing in the library depends on it.
void note_launch();

constexpr int kMaxDevices = 64;   // devices whose properties are looked up once

// Launch of a kernel that calls pdl_wait() (lg_common.cuh) before it touches global memory (or
// only for a hint, as the decode does): with `overlap` it may
// start while the kernel before it on the stream drains.  A failed launch is reported by the result alone: it does not
// stay behind as the runtime's last error, which a later call would take for its own.
template <typename... Params, typename... Args>
inline cudaError_t launch_clusters(bool overlap, int cluster_y, void (*kern)(Params...), dim3 grid, int block, int smem, cudaStream_t stream,
                                   const Args&... args) {
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (overlap) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster_y > 1) {   // clusters of 1 x cluster_y CTAs
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = attr[n].val.clusterDim.z = 1;
    attr[n++].val.clusterDim.y = static_cast<unsigned>(cluster_y);
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid; cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem; cfg.stream = stream;
  cfg.attrs = attr; cfg.numAttrs = n;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...);
  if (e == cudaSuccess) note_launch();
  else cudaGetLastError();
  return e;
}

template <typename... Params, typename... Args>
inline cudaError_t launch_kernel(bool overlap, void (*kern)(Params...), dim3 grid, int block, int smem, cudaStream_t stream, const Args&... args) {
  return launch_clusters(overlap, 1, kern, grid, block, smem, stream, args...);
}

// The same for a kernel that needs more dynamic shared memory than a launch may ask for by default (allowed once per
// device; a call on every launch cost the host a microsecond).
template <typename... Params, typename... Args>
inline cudaError_t launch_big_smem_clusters(bool overlap, int cluster_y, std::atomic<bool>* allowed /* [kMaxDevices] of this kernel */, void (*kern)(Params...), dim3 grid,
                                   int block, int smem, cudaStream_t stream, const Args&... args) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool known = dev < kMaxDevices && allowed[dev].load(std::memory_order_acquire);
  if (known && launch_clusters(overlap, cluster_y, kern, grid, block, smem, stream, args...) == cudaSuccess) return cudaSuccess;
  // (a device that was reset has forgotten it)
  if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess) { cudaGetLastError(); return e; }
  if (dev < kMaxDevices) allowed[dev].store(true, std::memory_order_release);
  return launch_clusters(overlap, cluster_y, kern, grid, block, smem, stream, args...);
}
template <typename... Params, typename... Args>
inline cudaError_t launch_big_smem(bool overlap, std::atomic<bool>* allowed, void (*kern)(Params...), dim3 grid, int block, int smem, cudaStream_t stream,
                                   const Args&... args) {
  return launch_big_smem_clusters(overlap, 1, allowed, kern, grid, block, smem, stream, args...);
}

struct Resolved {          // validated, defaulted copy of lg_attn_params
  int B, Hq, Hkv, L, D, block, mode, G;
  PatternDev pat;
  float scale;
  int exact_w;             // token-exact window length in tokens (0: block-granular)
  int win_block, win_phase;  // forward only, with exact_w: block-aligned window edge in coordinates shifted by win_phase (0: off)
  int64_t qs[3], ks[3], vs[3], os[3];
  int n_qtiles, n_ktiles;  // ceil(L / 128)
  int n_stiles, st_row0;   // super-tiles of the forward (256 rows each), and the pattern row the first one starts at
  int q_start, Lq;         // forward only: queries exist for rows [q_start, q_start + Lq) (0, L by default)
  const int32_t* doc_start;  // device [B, L] or null: first position of each token's document
  unsigned int* error_word;  // status word of the call when it is not the start of `ws` (null: it is)
  int lists_prepared;        // the caller says the workspace already holds this pattern's lists
  unsigned long long expect_fp, expect_fp2;   // fingerprints the kernels accept in the header (0: no check)
  int64_t nnz;
  int kv_total;              // kv heads (times batch) of the whole problem: B * Hkv, more when the call works a group of its heads
  KvSplit split;             // how the dK/dV pass cuts its kv tiles (calls with a backward; see kv_split)
  FwdSplit fsplit;           // which super-tiles the forward cuts (see fwd_split)
};

// want_bwd: the call runs, prepares or sizes a backward; kv_total: kv heads of the whole problem when `p` is a group of
// them (0: p is the whole)
lg_status resolve(const lg_attn_params* p, Resolved* r, bool want_bwd = false, int kv_total = 0);

// Layout of the attention workspace (all offsets 256-byte aligned).
struct WsLayout {
  // per schedule: start of each tile's entries, their number, the entries, by launch rank a TileRec of the tile
  size_t sq_off, sq_cnt, sq_ent, sq_order;       // super-tiles (forward)
  size_t qt_off, qt_cnt, qt_ent, qt_order;       // query tiles (dQ pass: over kv blocks, or over the kept dS tiles)
  size_t kt_off, kt_cnt, kt_ent, kt_order;       // kv tiles (dK/dV pass)
  size_t kt_cols;                                // pattern columns of each kv tile
  size_t doc_end;                                // int32 [B, L]: end of each token's document (bwd with documents only)
  size_t delta;                                  // 2 x float [B, Hq, L]: -LSE * log2 e, then -delta (bwd only)
  size_t ds_buf;                                 // dS^T tiles (backward that keeps dS only, 0 otherwise)
  size_t kv_part, kv_ticket;                     // dK/dV pass with split kv tiles: partial sums, arrivals per tile
  size_t total;
};
WsLayout ws_layout(const Resolved& r, bool want_bwd);

// Build CSR/CSC on `stream` into the given device arrays.
lg_status launch_index_build(const Resolved& r, int32_t* row_ptr, int32_t* col_idx, int32_t* col_ptr,
                             int32_t* row_idx, cudaStream_t stream);
struct RingCopy;
// Build the tile schedules inside a workspace.  `what`: bit 0 = the forward's schedule, bit 1 = the backward's
// schedules; `begin`: also reset the workspace's header first; `fp`: fingerprint to leave in it (0: none);
// `copy`: a ring to linearise in the same launch (null: none).
lg_status prepare_workspace(const Resolved& r, const WsLayout& w, uint8_t* ws, int what, bool begin,
                            unsigned long long fp, cudaStream_t stream, const RingCopy* copy = nullptr);

// bf16 [B, H, L, D] tensor (element strides bs, hs, ls; D contiguous) as a 4-D tensor map with
// boxes of 64 columns x `box_rows` rows and the 128-byte swizzle.
lg_status make_tmap(CUtensorMap* out, const void* base, int B, int H, int L, int D, const int64_t strides[3],
                    int box_rows);

// Which backward runs for this problem.
enum BwdVariant {
  kBwdTwoPass = 0,   // dK/dV pass, then a dQ pass that recomputes S and dP
  kBwdKeepDs = 2     // dK/dV pass that also writes dS^T to the workspace, then a dQ pass that is one product: dQ = dS K
};
BwdVariant bwd_variant(const Resolved& r);
// bytes of the dS^T buffer of the kBwdKeepDs variant
int sm_count();   // SMs of the current device, < 0 on failure
int head_group(const Resolved& r, int n_x);
size_t ds_buffer_bytes(const Resolved& r);


// Whether the attention kernels of a problem are launched overlapped: up to two forward CTAs per SM.  Their prologues
// and launch latencies then weigh something (2 heads x 512 tokens fwd + bwd 36.9 -> 35.9 us, steps of 40-50 us by
// 4-18 %).  Large ones gain nothing and lose 1-2 % (full causal, 32 heads x 16K: 8.55 -> 8.63 ms): CTAs that
// arrive as SMs fall free are spread over the chip in another order than those of an ordinary launch.
inline bool launch_attn_overlapped(const Resolved& r) {
  return static_cast<long long>(r.B) * r.Hq * r.n_stiles <= 2 * kSms;
}

// Which form of the forward a D = 64 problem takes (lg_fwd.cuh; both give the same bits).  Two CTAs on an SM hide each
// other's latencies, but one of them alone is 1.3-1.4 times as slow as the form that has the SM to itself, so they need
// a grid that keeps the pairs together until near its end.  Rounds of one CTA per SM from which the pairs are
// faster, measured over 230 problems of 8 to 7552 CTAs (time of the single form over that of the pairs):
//   rows of up to 512 keys on average       1.25   (208 CTAs 1.05-1.08, 128 CTAs 0.80-0.90)
//   up to 1152                              2      (window 1024: 416-528 CTAs 1.00-1.05, 128 CTAs 0.77-0.82)
//   longer rows                             4      (windows 2500-4096: 388-592 CTAs 0.91-1.00, 620-2048 CTAs 1.00-1.11)
//   full causal, lengths from 1 to L / 128  16     (1024 CTAs 0.89-0.95, 2048 CTAs 0.98-1.03, 4096 and more 1.00-1.13)
// 4 heads x 3318 tokens, full causal, 52 CTAs: 74 us in pairs, 53 us alone; 3 x 16 heads x 6001, window 1024, 1152 CTAs:
// 148 us in pairs, 164 us alone.
inline bool fwd_two_ctas(const Resolved& r) {
  if (r.D != 64) return false;
  const int64_t ctas = static_cast<int64_t>(r.B) * r.Hq * r.n_stiles, keys = r.nnz * r.block / r.pat.nB;
  const int quarter_rounds = r.mode == LG_MODE_FULL_CAUSAL ? 64 : keys > 1152 ? 16 : keys > 512 ? 8 : 5;
  return 4 * ctas > quarter_rounds * static_cast<int64_t>(kSms);
}

// Which tiles the forward of `r` cuts when the whole problem has `heads` query heads (times batch).  (Two CTAs on an SM: a
// grid of many rounds.  Documents: how long the tiles are is not known here, and pieces planned for tiles that are shorter
// cost more than they give: 4 heads x 8000 tokens in documents of 3000, full causal, 52 -> 60 us.)
inline FwdSplit fwd_split_of(const Resolved& r, int64_t heads) {
  Resolved whole = r;
  whole.B = 1;
  whole.Hq = static_cast<int>(heads);
  return r.doc_start || fwd_two_ctas(whole) ? FwdSplit{} : fwd_split(r.pat, r.D, r.st_row0, r.n_stiles, heads);
}

lg_status check_arch();
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

lg_status launch_fwd(const Resolved& r, const WsLayout& w, const void* q, const void* k, const void* v, void* o,
                     float* lse, uint8_t* ws, cudaStream_t stream);
lg_status launch_bwd(const Resolved& r, const WsLayout& w, const void* q, const void* k, const void* v,
                     const void* o, const float* lse, const void* d_o, void* dq, void* dk, void* dv, uint8_t* ws,
                     cudaStream_t stream, cudaEvent_t* marks /* null, or 4 events recorded around the 3 kernels */);

// The forward / backward entry points with the status word of the call redirected (null: the start
// of `workspace`): a step that runs several calls on slices of one workspace reports through one word.
lg_status attn_fwd_entry(const lg_attn_params* p, const void* q, const void* k, const void* v, void* o, float* lse,
                         void* workspace, size_t workspace_bytes, void* stream, unsigned int* status_word,
                         int kv_total = 0 /* kv heads of the whole problem when this is a group of them */);
lg_status attn_bwd_entry(const lg_attn_params* p, const void* q, const void* k, const void* v, const void* o,
                         const float* lse, const void* d_o, void* dq, void* dk, void* dv, void* workspace,
                         size_t workspace_bytes, void* stream, cudaEvent_t* marks, unsigned int* status_word,
                         int kv_total = 0 /* the same */);
size_t attn_workspace_bytes(const lg_attn_params* p, int want_bwd, int kv_total);

}  // namespace lg
