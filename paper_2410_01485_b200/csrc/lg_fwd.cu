// Launch of the forward attention kernel.
#include "lg_fwd.cuh"
#include "lg_host.h"

namespace lg {

template <int D, int BS, int NB, bool kSplit>
static lg_status launch_fwd_t(const Resolved& r, const WsLayout& w, const void* q, const void* k, const void* v,
                              void* o, float* lse, uint8_t* ws, cudaStream_t stream) {
  CUtensorMap tq, tk, tv;
  lg_status s;
  if ((s = make_tmap(&tq, q, r.B, r.Hq, r.Lq, D, r.qs, 128)) != LG_OK) return s;
  if ((s = make_tmap(&tk, k, r.B, r.Hkv, r.L, D, r.ks, BS)) != LG_OK) return s;
  if ((s = make_tmap(&tv, v, r.B, r.Hkv, r.L, D, r.vs, BS)) != LG_OK) return s;
  FwdArgs a;
  a.tile_ent = reinterpret_cast<const int32_t*>(ws + w.sq_ent);
  a.order = reinterpret_cast<const TileRec*>(ws + w.sq_order);
  a.o = static_cast<__nv_bfloat16*>(o);
  a.lse = lse;
  a.error_word = r.error_word ? r.error_word : reinterpret_cast<unsigned int*>(ws);
  a.expect_fp = r.expect_fp;
  a.n_tiles = r.n_stiles; a.nB = r.pat.nB; a.n_list = static_cast<int>(r.nnz);
  a.expect_fp2 = r.expect_fp2;
  for (int i = 0; i < 3; ++i) a.o_strides[i] = r.os[i];
  a.L = r.L; a.Hq = r.Hq; a.G = r.G;
  a.q_start = r.q_start; a.Lq = r.Lq;
  a.row_origin = r.st_row0 * r.block;
  a.exact_w = r.exact_w; a.ns = r.pat.ns;
  a.win_block = r.win_block; a.win_phase = r.win_phase;
  a.doc_start = r.doc_start;
  a.scale_log2 = r.scale * 1.4426950408889634f;
  a.head_group = head_group(r, r.B * r.Hq);
  a.split = r.fsplit;
  auto kern = fwd_kernel<D, BS, NB, kSplit>;
  constexpr int smem = FwdSmem<D>::kTotal;
  static std::atomic<bool> allowed[kMaxDevices];
  // cut tiles: clusters of as many CTAs as a tile has places; the last cluster is filled up
  const int cluster = kSplit ? r.fsplit.places : 1;
  const int n_y = r.n_stiles + (kSplit ? r.fsplit.n_cut * (cluster - 1) : 0);
  const dim3 grid(r.B * r.Hq, (n_y + cluster - 1) / cluster * cluster);
  return launch_big_smem_clusters(launch_attn_overlapped(r), cluster, allowed, kern, grid, kFwdThreads, smem, stream, tq, tk, tv, a) == cudaSuccess ? LG_OK : LG_ERR_CUDA;
}

lg_status launch_fwd(const Resolved& r, const WsLayout& w, const void* q, const void* k, const void* v, void* o,
                     float* lse, uint8_t* ws, cudaStream_t stream) {
  if (r.n_qtiles > 65535) return LG_ERR_UNSUPPORTED;
  const bool pairs = fwd_two_ctas(r);
#define LG_FWD_CASE(DD, BB, NN) \
  if (r.D == DD && r.block == BB && pairs == (NN == 1)) return launch_fwd_t<DD, BB, NN, false>(r, w, q, k, v, o, lse, ws, stream);
  // (where a part of a device cannot hold a cluster the launch is refused, and the tiles stay whole)
#define LG_FWD_CUT_CASE(DD, BB) \
  if (r.fsplit.len > 0 && r.D == DD && r.block == BB && launch_fwd_t<DD, BB, 2, true>(r, w, q, k, v, o, lse, ws, stream) == LG_OK) return LG_OK;
  LG_FWD_CUT_CASE(128, 128)
  LG_FWD_CUT_CASE(128, 64)
  LG_FWD_CUT_CASE(64, 128)
  LG_FWD_CUT_CASE(64, 64)
#undef LG_FWD_CUT_CASE
  LG_FWD_CASE(128, 128, 2)
  LG_FWD_CASE(128, 64, 2)
  LG_FWD_CASE(64, 128, 1)
  LG_FWD_CASE(64, 128, 2)
  LG_FWD_CASE(64, 64, 1)
  LG_FWD_CASE(64, 64, 2)
#undef LG_FWD_CASE
  return LG_ERR_UNSUPPORTED;
}

}  // namespace lg
