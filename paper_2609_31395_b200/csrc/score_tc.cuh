// Tensor-core path of actkv_score for sm_100a: tcgen05.mma with TMEM accumulators, operands
// staged by TMA (cp.async.bulk.tensor, 128-byte swizzle) straight from the paged pool through the
// block table, one TMA box per (page, half of the head dimension).
//
// Two kernels, both warp-specialised (warp 0: TMA producer, warp 1: MMA issuer + TMEM owner,
// the other warps: epilogue reading TMEM with tcgen05.ld):
//
//  * LSE pass (score_tc_lse.cuh; Section 7.1, LSE equation).  D[row, key] = Q K^T with the window x
//    group rows on the TMEM lanes (Q as the A operand from tensor memory), so every epilogue thread
//    owns one row per 128-row block and keeps its running (reference, sum of exp2): no shuffles.
//  * Pooled-score pass (score_tc_pool.cuh; Section 7.1 recovery identity, Algorithm 3 steps 3-5).
//    The transposed product D[key, row] = K Q^T with the keys on the lanes and row = w*G + g on the
//    columns, so the max over the GQA group and the sum over the action tokens run inside one
//    thread.  Because exp is monotone the max over the group is taken on (s - lse) BEFORE the exp:
//    W exps per key instead of W*G.
//
// Every wait on an mbarrier is bounded (wall-clock limit); on give-up the kernel records
// ACTKV_E_TIMEOUT in the status word, every role leaves its loop, outstanding MMAs are drained,
// TMEM is freed and the CTA returns.
//
// This file: tensor-map creation and launch configuration (host side).
#pragma once

#include <algorithm>
#include <atomic>

#include "score_tc_lse.cuh"
#include "score_tc_pool.cuh"

namespace actkv {
namespace tc {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver entry point is looked up through the runtime, so the library does not link libcuda.
inline EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = []() -> EncodeTiledFn {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    return (EncodeTiledFn)p;
  }();
  return fn;
}

// The four-dimensional K map needs the slots of consecutive pages to continue at the slot stride.
inline bool pool_needs_5d(const actkv_pool_t* pool) { return pool->stride_page != (int64_t)pool->page_size * pool->stride_slot; }

inline int pow2_at_least(int g) { int p = 1; while (p < g) p <<= 1; return p; }

// CTAs per unit for a launch over `units` units of `tiles` key tiles each.  One CTA is resident per SM, so a
// launch runs in rounds of 148 CTAs and the last round is partly empty; more CTAs make that round
// cheaper, but every CTA pays a fixed cost (operand set-up, pipeline fill and drain) of about `ovh` key
// tiles' worth.  Returns the count in [1, n_max] with the best product of the two, preferring fewer CTAs
// unless more are clearly better.
inline int best_split(int64_t units, int tiles, int ovh, int n_max) {
  int best = 1;
  double best_eff = 0.0;
  if (units < 1) units = 1;
  for (int n = 1; n <= n_max; ++n) {
    const int tpc = (tiles + n - 1) / n;
    if (tpc < 1) break;
    const int64_t grid = units * ((tiles + tpc - 1) / tpc);
    const int64_t rounds = (grid + 147) / 148;
    const double eff = (double)grid / (double)(rounds * 148) * (double)tpc / (double)(tpc + ovh);
    if (eff > best_eff * 1.005) { best_eff = eff; best = n; }
  }
  return best;
}

// What a work item of the LSE pass costs beside its key tiles, in tiles (Q blocks into tensor memory, references, merge): 4 K cycles; 8 K
// where its Q blocks wait for the columns of the item before (measured from job to job: 2157 cycles a tile of two blocks in whole units, 2423
// on average in eight chunks; three blocks 2255 x 1.5, and 2615 x 1.5).
inline double lse_item_overhead(int rows, int head_dim) {
  return rows <= 128 ? 3.0 : rows > 256 && rows <= 384 && head_dim == 128 ? 2.8 : 2.0;
}

// Share of a last item by which launches of unequal requests end late: half of one of two blocks, and as many jobs of one of three.
inline double lse_tail(int rows) { return rows > 256 && rows <= 384 ? 0.75 : 0.5; }

// Chunks per unit of the LSE pass, whose CTAs go on from item to item, for a launch over `units` units of `tiles` key tiles, an item costing
// its tiles and `ovh` more.  Equal units run in rounds of 148 of which the last is partly empty; requests of different lengths or windows
// (mean over longest: `len`, `win`) spread evenly but for the last items, half of one on average, once there are more items than SMs.
// Returns the count in [1, n_max] that costs least, preferring fewer unless more are clearly better.
// 8 layers x 8 heads, 4 requests of 6500-15000 keys, head_dim 64, 200-512 rows: 410 us with whole units, 341 with the three chunks this
// gives (four 336, five 334, eight 344).  4 layers x 8 heads, 4 x 16000 keys, 192 rows: 148 us with whole units, 158 with eight chunks (half
// a percent in the model decided for those before).
inline int lse_split(int64_t units, int tiles, double len, double win, double ovh, double tail, int n_max) {
  const bool equal = len > 0.999 && win > 0.999;
  int best = 1;
  double best_t = 1e300;
  for (int n = 1; n <= n_max; ++n) {
    const int tpc = (tiles + n - 1) / n;
    if (tpc < 4 && n > 1) break;
    const int64_t items = units * ((tiles + tpc - 1) / tpc);
    double t;
    if (equal) t = (double)((items + 147) / 148) * (tpc + ovh);
    else if (items <= 148) t = tpc + ovh;
    else t = ((double)units * tiles * len * win + (double)items * len * ovh) / 148.0 + tail * (tpc + ovh);
    if (t < best_t * (equal ? 0.99 : 0.995)) { best_t = t; best = n; }
  }
  return best;
}

inline bool make_kmap(const actkv_pool_t* pool, CUtensorMap* kmap) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return false;
  // K half of the pool.  Slot-major pages whose slots continue across pages: [layer][slot (page*16 + s)]
  // [head][dim], four dimensions (measured 13 % faster than five on the K stream).  Any other page layout
  // (head-major pages): [layer][page][head][slot][dim] with the caller's strides.  A box is one page of
  // one head, 64 dims: page_size rows of 128 B.
  CUresult res;
  if (!pool_needs_5d(pool)) {
    cuuint64_t dims[4] = {(cuuint64_t)pool->head_dim, (cuuint64_t)pool->n_kv_heads, (cuuint64_t)pool->n_pages * pool->page_size,
                          (cuuint64_t)pool->n_layers};
    cuuint64_t strides[3] = {(cuuint64_t)pool->stride_head * 2, (cuuint64_t)pool->stride_slot * 2,
                             (cuuint64_t)pool->stride_layer * 2};
    cuuint32_t box[4] = {64, 1, (cuuint32_t)pool->page_size, 1};
    cuuint32_t es[4] = {1, 1, 1, 1};
    res = enc(kmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, pool->base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  } else {
    cuuint64_t dims[5] = {(cuuint64_t)pool->head_dim, (cuuint64_t)pool->page_size, (cuuint64_t)pool->n_kv_heads,
                          (cuuint64_t)pool->n_pages, (cuuint64_t)pool->n_layers};
    cuuint64_t strides[4] = {(cuuint64_t)pool->stride_slot * 2, (cuuint64_t)pool->stride_head * 2,
                             (cuuint64_t)pool->stride_page * 2, (cuuint64_t)pool->stride_layer * 2};
    cuuint32_t box[5] = {64, (cuuint32_t)pool->page_size, 1, 1, 1};
    cuuint32_t es[5] = {1, 1, 1, 1, 1};
    res = enc(kmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, pool->base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  }
  return res == CUDA_SUCCESS;
}

// q: [slab*sum_win + w][q head][head_dim]; a box is (64 dims, `heads` heads from the first of a group on, `tokens` window tokens)
inline bool make_qmap(const actkv_pool_t* pool, const void* q, int nls, int sum_win, int n_q_heads, int heads, int tokens,
                      CUtensorMap* qmap) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return false;
  const cuuint64_t D = (cuuint64_t)pool->head_dim;
  cuuint64_t dims[3] = {D, (cuuint64_t)n_q_heads, (cuuint64_t)nls * sum_win};
  cuuint64_t strides[2] = {D * 2, (cuuint64_t)n_q_heads * D * 2};
  cuuint32_t box[3] = {64, (cuuint32_t)heads, (cuuint32_t)tokens};
  cuuint32_t es[3] = {1, 1, 1};
  return enc(qmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(q), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Fault-injection hook of the bounded waits (actkv_debug_inject_stall): while stall_tile >= 0 the K-tile
// producers of every tensor-core score launch issue no tile from that one on, and every wait gives up after
// `wait_cycles`.  Process-wide, read at launch.
struct StallHook {
  std::atomic<int32_t> stall_tile{-1};
  std::atomic<long long> wait_cycles{WAIT_LIMIT_CYCLES};
};
inline StallHook& stall_hook() { static StallHook h; return h; }
inline void apply_hook(TcArgs& ta) {
  ta.stall_tile = stall_hook().stall_tile.load();
  ta.wait_cycles = stall_hook().wait_cycles.load();
}

}  // namespace tc

// The tensor-core path takes: pages of 16, 32, 64 or 128 tokens, head_dim 128 or 64, slot-major or head-major pages (any
// strides that are multiples of 16 bytes), 128-byte aligned base, group size <= 32 (padded to a power of two in the
// pooled-score pass), min_rows <= window x group rows <= 4096 (more than 512 are taken in groups: of 512 rows a launch in the
// pooled-score pass, of 256 an item in the LSE pass), positive softmax scale.
// The full score (LSE + pooled pass) takes it from 64 rows up; the streaming update, which runs the pooled pass alone and is
// bound by the K reads, from a single row.  The two families, us, 4 layers x 8 heads, 8 requests of 9000 keys, head_dim 128,
// group 4 (mma.sync beyond 48 rows on a pool 16 bytes off the 128-byte boundary, which costs it up to a quarter):
//   rows             16         32         48         64         96
//   LSE, mma / tc    118 / -    135 / -    159 / -    206 / 163  356 / 164
//   pooled, mma / tc 107 / 119  131 / 121  163 / 121  212 / 122  367 / 127
// so the LSE passes meet around 48 rows, and one line for both passes is late for the pooled one.  head_dim 64, group 8, 8
// layers: LSE 170 at 48 rows, 204 / 228 at 64, 337 / 230 at 96.
inline bool score_tc_supported(const actkv_pool_t* p, int G, int max_win, float sm_scale, const void* q,
                               int min_rows = 64) {
  if (p->page_size != 16 && p->page_size != 32 && p->page_size != 64 && p->page_size != 128) return false;
  if (p->head_dim != 128 && p->head_dim != 64) return false;
  // TMA: every stride a positive multiple of 16 bytes (any page layout with contiguous head dimensions)
  if (p->stride_head <= 0 || p->stride_slot <= 0 || p->stride_page <= 0 || p->stride_layer <= 0) return false;
  if ((p->stride_head % 8) || (p->stride_slot % 8) || (p->stride_page % 8) || (p->stride_layer % 8)) return false;
  if (((uintptr_t)p->base & 127) || ((uintptr_t)q & 127)) return false;
  if (G < 1 || G > 32) return false;
  if (max_win * G < min_rows) return false;
  const int rows = max_win * tc::pow2_at_least(G);     // rows of the pooled-score pass (groups padded to a power of two)
  if (rows > tc::MAX_ROWS_TOTAL) return false;
  if (!(sm_scale > 0.f)) return false;
  return tc::encode_fn() != nullptr;
}

template <int NH, bool REGS>
inline int score_tc_launch_lse_c(const CUtensorMap& kmap, const CUtensorMap& qmap, const tc::TcArgs& ta, unsigned grid, cudaStream_t s) {
  constexpr int NPOLY = tc::LSE_NPOLY;
  const size_t smem = (size_t)tc::lse_stages(NH) * NH * tc::HALF_BYTES + sizeof(tc::LseBarriers);
  auto kern = ta.a.win_left > 0 ? tc::score_tc_lse_kernel<NPOLY, NH, true, REGS> : tc::score_tc_lse_kernel<NPOLY, NH, false, REGS>;
  if (ensure_dyn_smem(kern, smem) != cudaSuccess) return ACTKV_E_CUDA;
  launch_pdl(kern, grid, tc::LSE_THREADS, smem, s, kmap, qmap, ta, tc::Exp2Cubic{tc::EXP2_C0, tc::EXP2_C1, tc::EXP2_C2, tc::EXP2_C3});
  ACTKV_CHECK_LAUNCH();
  return ACTKV_OK;
}

inline int score_tc_launch_lse(ScoreArgs& a, const actkv_pool_t* pool, int max_win, cudaStream_t s) {
  CUtensorMap kmap, qmap;
  if (!tc::make_kmap(pool, &kmap) ||
      !tc::make_qmap(pool, a.q, a.n_layers_sub, a.sum_win, a.n_q_heads, a.group, 64 / a.group, &qmap))
    return ACTKV_E_CUDA;
  tc::TcArgs ta;
  ta.a = a;
  ta.n_rg = tc::lse_row_groups(max_win * a.group);
  ta.row_begin = 0;
  ta.k5 = tc::pool_needs_5d(pool) ? 1 : 0;
  ta.n_stages = 0;
  ta.tiles_per_cta = 0;
  ta.n_kchunks = 0;
  ta.copy_ws = nullptr;              // (this kernel has no copy role)
  tc::apply_hook(ta);
  const int64_t units = (int64_t)a.n_layers_sub * a.pool.n_kv_heads * a.tab.n_req;
  const int64_t grid = units * a.n_chunks * ta.n_rg;
  if (grid > 0x7fffffffLL) return ACTKV_E_INVALID;
  const bool regs = tc::lse_moves(max_win * a.group);
  if (pool->head_dim == 64)
    return regs ? score_tc_launch_lse_c<1, true>(kmap, qmap, ta, (unsigned)grid, s) : score_tc_launch_lse_c<1, false>(kmap, qmap, ta, (unsigned)grid, s);
  return regs ? score_tc_launch_lse_c<2, true>(kmap, qmap, ta, (unsigned)grid, s) : score_tc_launch_lse_c<2, false>(kmap, qmap, ta, (unsigned)grid, s);
}

template <int G>
inline int score_tc_launch_pool_g(const CUtensorMap& kmap, const CUtensorMap& qmap, const tc::TcArgs& ta, bool aug, unsigned grid,
                                  size_t smem, cudaStream_t s) {
  const bool d64 = ta.a.pool.head_dim == 64;
  auto kern = d64 ? tc::score_tc_pool_kernel<G, 1, false> : tc::score_tc_pool_kernel<G, 2, false>;
  if constexpr (tc::aug_group(G))
    if (aug) kern = d64 ? tc::score_tc_pool_kernel<G, 1, true> : tc::score_tc_pool_kernel<G, 2, true>;
  // The warpgroups of this kernel re-divide the registers the launch allocates; the epilogue warpgroups would
  // wait for ever for registers that a smaller allocation does not have, so the allocation is checked first.
  if (kernel_num_regs(kern) < tc::POOL_REGS_ENTRY) return ACTKV_E_CUDA;
  if (ensure_dyn_smem(kern, smem) != cudaSuccess) return ACTKV_E_CUDA;
  launch_pdl(kern, grid, tc::POOL_THREADS, smem, s, kmap, qmap, ta);
  ACTKV_CHECK_LAUNCH();
  return ACTKV_OK;
}

inline int score_tc_launch_score(ScoreArgs& a, const actkv_pool_t* pool, int max_tok, int max_win, cudaStream_t s,
                                 CompactWs* copy_ws) {
  CUtensorMap kmap, qmap;
  const int Gp = tc::pow2_at_least(a.group);       // (this kernel pads a group to a power of two)
  if (!tc::make_kmap(pool, &kmap) || !tc::make_qmap(pool, a.q, a.n_layers_sub, a.sum_win, a.n_q_heads, Gp, 128 / Gp, &qmap))
    return ACTKV_E_CUDA;
  tc::TcArgs ta;
  ta.a = a;
  const int rows_all = max_win * Gp;
  const int nh = pool->head_dim / 64;
  const int rows_pad = (std::min(rows_all, tc::MAX_ROWS) + 127) & ~127;      // of the largest unit, per launch
  const int n_rc = (rows_pad + 255) / 256;
  // Every unit lays out its own shared memory: the widest one must have its queries and POOL_MIN_STAGES key tiles,
  // everyone takes what is left for more of them.
  // (the kernel without the LSE in the contraction when no unit would use it: few rows, a group it is not done for, or every
  // window as long as the longest and that beyond the limit; or when dividing by the scale could overflow)
  const bool aug = rows_all > 64 && tc::aug_group(Gp) && a.scale_log2 >= 1e-30f && !(rows_all > tc::aug_rows(nh) && (int64_t)a.sum_win == (int64_t)a.tab.n_req * max_win);
  const size_t fixed = (size_t)n_rc * nh * tc::QBLK_BYTES + tc::POOL_FIXED;
  const size_t tables = aug && rows_pad <= tc::aug_rows(nh) ? tc::AUG_K_BYTES + (size_t)n_rc * tc::AUG_CHUNK_BYTES : 0;
  ta.n_stages = (int32_t)std::min<size_t>(tc::POOL_STAGES, (tc::SMEM_LIMIT - fixed) / (nh * tc::HALF_BYTES));
  if (fixed + tables + tc::POOL_MIN_STAGES * nh * tc::HALF_BYTES > tc::SMEM_LIMIT) return ACTKV_E_INVALID;
  ta.n_rg = 0;
  ta.k5 = tc::pool_needs_5d(pool) ? 1 : 0;
  ta.copy_ws = copy_ws;
  tc::apply_hook(ta);
  const int64_t units = (int64_t)a.n_layers_sub * a.pool.n_kv_heads * a.tab.n_req;
  const int max_tiles = (max_tok + tc::TK - 1) / tc::TK;
  // CTAs per unit: one CTA per SM is resident, so the launch runs in rounds of 148 CTAs and the last round
  // is partly empty; more CTAs make that round cheaper, but every CTA pays for its Q load and its pipeline
  // fill (about three key tiles' worth).  Take the count with the best product of the two, of ranges of two key tiles and more
  // (that few only where SMs would stay idle).
  ta.n_kchunks = tc::best_split(units, max_tiles, 3, std::min(64, std::max(1, max_tiles / 2)));
  ta.tiles_per_cta = (max_tiles + ta.n_kchunks - 1) / ta.n_kchunks;
  ta.n_kchunks = (max_tiles + ta.tiles_per_cta - 1) / ta.tiles_per_cta;
  const int64_t grid = units * ta.n_kchunks;
  if (grid > 0x7fffffffLL) return ACTKV_E_INVALID;
  const size_t smem = tc::SMEM_LIMIT;
  // a window of more than MAX_ROWS rows: one launch per group of MAX_ROWS rows (whole action tokens), in
  // stream order; the first writes the score, the others add their share of the mean
  for (int row_begin = 0; row_begin < rows_all; row_begin += tc::MAX_ROWS) {
    ta.row_begin = row_begin;
    int rc = ACTKV_E_INVALID;
    switch (Gp) {
      case 1: rc = score_tc_launch_pool_g<1>(kmap, qmap, ta, aug, (unsigned)grid, smem, s); break;
      case 2: rc = score_tc_launch_pool_g<2>(kmap, qmap, ta, aug, (unsigned)grid, smem, s); break;
      case 4: rc = score_tc_launch_pool_g<4>(kmap, qmap, ta, aug, (unsigned)grid, smem, s); break;
      case 8: rc = score_tc_launch_pool_g<8>(kmap, qmap, ta, aug, (unsigned)grid, smem, s); break;
      case 16: rc = score_tc_launch_pool_g<16>(kmap, qmap, ta, aug, (unsigned)grid, smem, s); break;
      case 32: rc = score_tc_launch_pool_g<32>(kmap, qmap, ta, aug, (unsigned)grid, smem, s); break;
      default: break;
    }
    if (rc != ACTKV_OK) return rc;
  }
  return ACTKV_OK;
}

}  // namespace actkv
