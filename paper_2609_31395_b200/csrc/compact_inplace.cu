// actkv_compact_inplace: in-place compaction into the last X logical blocks of every request
// (Section 7.2 region equations; Algorithm 4), one keep mask per (layer, KV head).
//
// For a request with L used slots in Y = ceil(L/BS) blocks and budget B < L:  X = ceil(B/BS),
// Start = (Y-X)*BS, End = Start + B.  Holes of the region (slots of [Start, End) that are not kept,
// including allocated-but-unused slots past L) are the destinations, survivors outside the region are
// the sources, both in ascending order, zipped.  With the keep mask given as the ascending index list
// sel[0..B) the plan needs no scan and no scratch:
//     a = #kept below Start, c = #kept below End,
//     hole p has rank j = (p - Start) - (#kept in [Start, p)),
//     its source is the j-th survivor outside the region: sel[j] if j < a, else sel[c + j - a].
// Two kernels on one stream:
//   copy     : one CTA per (run of region slots, request, layer x head): the kept ones are marked in a
//              bitmap, every other slot finds its rank and source, the CTA's moves are packed in
//              shared memory and copied as 16-byte vectors, several loads in flight per thread.
//              Sources lie outside the region and destinations inside it, so one pass is conflict-free.
//   finalize : page_table[r] <- its last X pages, seq_len[r] <- B, the first Y-X pages are pushed on
//              the free-list stack (only on the call whose layer range ends at the pool's last layer).
// On a device-detected error the tables stay as they were; only dead slots (holes) were written.
// The copy can also be deferred (actkv_compact_inplace_begin / _end): the moves of a layer group are resolved
// once into a table of (source, destination) row offsets, 32 region slots per item, and published as the work
// queue of compact_job.cuh, so that the spare warps of the pooled-score kernel of the NEXT layer group execute
// them (sources and destinations lie in layers that kernel does not touch) and a drain kernel what is left.
#include "compact_job.cuh"
#include "warp_search.cuh"

namespace actkv {

constexpr int CI_UNROLL = 8;

__device__ __forceinline__ int lower_bound_i32(const int32_t* __restrict__ a, int n, int32_t key) {
  int lo = 0, hi = n;                                        // first index with a[idx] >= key
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (a[mid] < key) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// The same by one converged warp, 32 probes at a time: four round trips to memory for 64 K entries instead of sixteen.
__device__ __forceinline__ int warp_lower_bound_i32(const int32_t* __restrict__ a, int n, int32_t key) {
  const int lane = threadIdx.x & 31;
  SearchSpan s{0, n};
  while (s.hi - s.lo > 32) {
    const int probe = search_probe(s, lane);
    s = search_narrow(s, __popc(__ballot_sync(0xffffffffu, probe < s.hi && a[probe] < key)));
  }
  return s.lo + __popc(__ballot_sync(0xffffffffu, s.lo + lane < s.hi && a[s.lo + lane] < key));
}

// A CTA of NT threads takes PER * NT slots of the region.  The kept slots among them are marked in a bitmap (they are
// consecutive entries of the list), so that a slot knows from it whether it is a hole and which one.
// What bounds it: the copies, once the searches at the start are few and short.  With 128 slots per CTA and
// binary searches, a CTA spent most of its life in fourteen
// dependent loads: 8 layers x 8 heads, 16 requests of 8K-24K tokens, 80 % kept, 724 us, now 454 (2.6 GB, 5.7 TB/s); half
// kept 710 -> 625 us (4.0 GB, 6.4 TB/s).
template <int VPR_SHIFT, int NT, int PER>
__global__ void __launch_bounds__(NT) compact_inplace_copy_kernel(
    PoolView pool, TablesView tab, int32_t layer_begin, const int32_t* __restrict__ sel_idx, int64_t sel_stride,
    const int32_t* __restrict__ keep_indptr, const int32_t* __restrict__ budget, int32_t max_keep,
    int32_t* __restrict__ new_order, int32_t* status) {
  pdl_begin(sel_idx, keep_indptr, budget);
  constexpr int SLOTS = NT * PER, WORDS = SLOTS / 32;
  __shared__ uint32_t s_kept[WORDS];                         // bitmap of the kept slots
  __shared__ int32_t s_before[WORDS];                        // kept slots in earlier words
  __shared__ int64_t s_src[SLOTS], s_dst[SLOTS];
  __shared__ int32_t s_a, s_c, s_lb0, s_cnt;

  const int r = blockIdx.y;
  const int H = pool.n_kv_heads, P = pool.page_size, D = pool.head_dim;
  const int slab = blockIdx.z / H, h = blockIdx.z - slab * H;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int32_t L = tab.seq_len[r], b_raw = budget[r], kept_off = keep_indptr[r];
  if (status_set(status)) return;
  const int32_t B = b_raw < 0 ? 0 : b_raw;
  const int32_t* sel = sel_idx + (int64_t)blockIdx.z * sel_stride + kept_off;
  int32_t* ord = new_order ? new_order + (int64_t)blockIdx.z * sel_stride + kept_off : nullptr;
  const int32_t i0 = blockIdx.x * SLOTS;                     // first region slot of this CTA, relative to Start

  if (B >= L) {                                              // not compacting: the order is the identity list
    if (ord)
      for (int i = i0 + tid; i < min(L, i0 + SLOTS); i += NT) ord[i] = sel[i];
    return;
  }
  if (i0 >= B) return;
  const int Y = (L + P - 1) / P, X = (B + P - 1) / P;
  if (Y > tab.max_pages || B > max_keep) {
    if (tid == 0) report(status, ACTKV_E_INVALID, r, Y > tab.max_pages ? L : B);
    return;
  }
  const int32_t start = (Y - X) * P, end = start + B;
  const int32_t p0 = start + i0;

  if (warp < 3) {
    const int v = warp_lower_bound_i32(sel, B, warp == 0 ? start : warp == 1 ? end : p0);
    if (lane == 0) (warp == 0 ? s_a : warp == 1 ? s_c : s_lb0) = v;
  }
  if (tid < WORDS) s_kept[tid] = 0u;
  if (tid == 96) s_cnt = 0;
  __syncthreads();
  const int a = s_a, c = s_c, lb0 = s_lb0;
  const int m = a + (B - c);                                 // survivors outside the region = holes inside it
  // at most SLOTS kept indices fall in this CTA's slots: they all sit in sel[lb0 .. lb0 + SLOTS)
  const int wn = min(SLOTS, B - lb0);
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int t = k * NT + tid;
    if (t < wn) {
      const int32_t x = sel[lb0 + t];
      // the list must be strictly ascending for the plan to be conflict-free
      if (t + 1 < wn) {
        const int32_t y = sel[lb0 + t + 1];
        if (y <= x) report(status, ACTKV_E_BADINDEX, r, y);
      }
      const int32_t d = x - p0;
      if (d >= 0 && d < SLOTS) atomicOr(&s_kept[d >> 5], 1u << (d & 31));
    }
  }
  __syncthreads();
  static_assert(WORDS <= 32, "one warp scans the bitmap");
  if (warp == 0) {
    const int v = lane < WORDS ? __popc(s_kept[lane]) : 0;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane < WORDS) s_before[lane] = incl - v;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int t = k * NT + tid;                              // (a warp's slots are one word of the bitmap)
    const int32_t p = p0 + t;
    bool hole = false;
    int32_t src_pos = -1;
    if (p < end) {
      const uint32_t word = s_kept[t >> 5];
      if ((word >> lane) & 1u) {
        if (ord) ord[p - start] = p;
      } else {
        const int w = s_before[t >> 5] + __popc(word & ((1u << lane) - 1u));       // #kept in [p0, p)
        const int j = (p - start) - (lb0 + w - a);           // rank of this hole
        if (j < 0 || j >= m) {
          report(status, ACTKV_E_BADINDEX, r, p);
        } else {
          src_pos = j < a ? sel[j] : sel[c + (j - a)];
          if ((uint32_t)src_pos >= (uint32_t)L || (src_pos >= start && src_pos < end)) {
            report(status, ACTKV_E_BADINDEX, r, src_pos);
          } else {
            hole = true;
            if (ord) ord[p - start] = src_pos;
          }
        }
      }
    }
    // a move whose source or destination page id is out of range is dropped (and reported): nothing is read
    // from or written to a page the request does not own
    int32_t sp = -1, dp = -1;
    if (hole) {
      sp = page_or_neg(tab, pool.n_pages, r, src_pos / P, status);
      dp = page_or_neg(tab, pool.n_pages, r, p / P, status);
      if (sp < 0 || dp < 0) hole = false;
    }
    // pack this CTA's moves (their order within the CTA does not matter)
    const uint32_t bal = __ballot_sync(0xffffffffu, hole);
    int wbase = 0;
    if (lane == 0 && bal) wbase = atomicAdd(&s_cnt, __popc(bal));
    wbase = __shfl_sync(0xffffffffu, wbase, 0);
    if (hole) {
      const int q = wbase + __popc(bal & ((1u << lane) - 1u));
      s_src[q] = (int64_t)sp * pool.stride_page + (int64_t)(src_pos % P) * pool.stride_slot + (int64_t)h * pool.stride_head;
      s_dst[q] = (int64_t)dp * pool.stride_page + (int64_t)(p % P) * pool.stride_slot + (int64_t)h * pool.stride_head;
    }
  }
  __syncthreads();
  const int cnt = s_cnt;
  __nv_bfloat16* lbase = const_cast<__nv_bfloat16*>(pool.base) + (int64_t)(layer_begin + slab) * pool.stride_layer;
  const int vpr = D / 8;
  const int per_kv = (VPR_SHIFT >= 0) ? (cnt << VPR_SHIFT) : cnt * vpr;
  const int total = 2 * per_kv;
  for (int v0 = tid; v0 < total; v0 += NT * CI_UNROLL) {
    uint4 val[CI_UNROLL];
    int64_t doff[CI_UNROLL];
#pragma unroll
    for (int k = 0; k < CI_UNROLL; ++k) {
      const int v = v0 + k * NT;
      doff[k] = -1;
      if (v < total) {
        const int kv = v >= per_kv ? 1 : 0;
        const int rem = v - kv * per_kv;
        const int i = (VPR_SHIFT >= 0) ? (rem >> VPR_SHIFT) : rem / vpr;
        const int dv = (VPR_SHIFT >= 0) ? (rem & ((1 << VPR_SHIFT) - 1)) : rem - i * vpr;
        const int64_t kvo = (int64_t)kv * pool.stride_kv + dv * 8;
        val[k] = *reinterpret_cast<const uint4*>(lbase + s_src[i] + kvo);
        doff[k] = s_dst[i] + kvo;
      }
    }
#pragma unroll
    for (int k = 0; k < CI_UNROLL; ++k)
      if (doff[k] >= 0) *reinterpret_cast<uint4*>(lbase + doff[k]) = val[k];
  }
}

// ---- deferred form --------------------------------------------------------------------------------
// Plan: items per request (32 region slots each; with an order output also the requests that are not
// compacted, whose order is the identity list), their prefix sums, and the job record.
__global__ void compact_inplace_plan_kernel(TablesView tab, PoolView pool, const int32_t* __restrict__ budget,
                                            int32_t max_keep, int32_t want_order, int32_t layer_begin, int32_t n_layers,
                                            int32_t vpr_shift, uint32_t* src_tab, uint32_t* dst_tab, int64_t tab_items,
                                            CompactWs* ws, int32_t* status) {
  pdl_begin(budget);
  if (threadIdx.x != 0) return;
  const int R = tab.n_req, P = pool.page_size;
  int32_t* item_off = ws_item_off(ws, R);
  bool ok = !status_set(status);
  int64_t off = 0;
  for (int r = 0; r < R; ++r) {
    item_off[r] = (int32_t)off;
    const int32_t L = tab.seq_len[r];
    const int32_t B = budget[r] < 0 ? 0 : budget[r];
    if (L < 0) { report(status, ACTKV_E_INVALID, r, L); ok = false; continue; }
    if (B >= L) {
      if (want_order) off += (L + 31) / 32;
      continue;
    }
    const int Y = (L + P - 1) / P;
    if (Y > tab.max_pages || B > max_keep) { report(status, ACTKV_E_INVALID, r, Y > tab.max_pages ? L : B); ok = false; continue; }
    off += (B + 31) / 32;
  }
  item_off[R] = (int32_t)off;
  const int64_t per_slab = off * pool.n_kv_heads;
  const int64_t items = per_slab * n_layers;
  if (items > 0x7fffffff || items > tab_items) {         // (the host sized the tables for max_keep)
    if (ok) report(status, ACTKV_E_WORKSPACE, -1, (int32_t)min(items, (int64_t)0x7fffffff));
    ok = false;
  }
  ws->plan_ok = ok ? 1 : 0;
  ws->total_new = (int32_t)off;                 // items of one (layer, head)
  ws->next_item = 0u;
  ws->n_items = ok ? (int32_t)items : 0;
  ws->pool = pool;
  ws->tab = tab;
  ws->sel_idx = nullptr;
  ws->sel_stride = 0;
  ws->keep_indptr = nullptr;
  ws->budget = budget;
  ws->status = status;
  ws->layer_begin = layer_begin;
  ws->n_layers = n_layers;
  ws->vpr_shift = vpr_shift;
  ws->parts_per_page = 1;
  ws->role_items = 0;
  ws->pad = CJ_INPLACE_MARK;
  ws->src_tab = src_tab;
  ws->dst_tab = dst_tab;
  ws->items_per_slab = (int32_t)max((int64_t)1, min(per_slab, (int64_t)0x7fffffff));
  ws->free_count = 0;
}

// One warp per item: the 32 region slots [32 chunk, 32 chunk + 32) of one (layer, head, request), classified as
// in the one-launch kernel above; a hole's move goes into the table as (source, destination) offsets in 16-byte
// units within the layer, everything else as CJ_NONE.
__global__ void __launch_bounds__(128) compact_inplace_resolve_kernel(
    CompactWs* ws, const int32_t* __restrict__ sel_idx, int64_t sel_stride, const int32_t* __restrict__ keep_indptr,
    int32_t* __restrict__ new_order) {
  pdl_begin(sel_idx, keep_indptr);
  const int lane = threadIdx.x & 31;
  const int64_t n = cj_count(ws);
  const PoolView& pool = ws->pool;
  const TablesView& tab = ws->tab;
  const int R = tab.n_req, H = pool.n_kv_heads, P = pool.page_size;
  const int32_t* item_off = ws_item_off(ws, R);
  const int per_head = ws->total_new, per_slab = ws->items_per_slab;
  int32_t* status = ws->status;
  for (int64_t item = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5); item < n; item += (int64_t)gridDim.x * 4) {
    const int slab = (int)(item / per_slab), rem = (int)(item - (int64_t)slab * per_slab);
    const int h = rem / per_head, rem2 = rem - h * per_head;
    int lo = 0, hi = R;                                  // item_off[lo] <= rem2 < item_off[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (item_off[mid] <= rem2) lo = mid; else hi = mid;
    }
    const int r = lo, chunk = rem2 - item_off[r];
    const int z = slab * H + h;
    const int32_t L = tab.seq_len[r];
    const int32_t B = ws->budget[r] < 0 ? 0 : ws->budget[r];
    const int32_t* sel = sel_idx + (int64_t)z * sel_stride + keep_indptr[r];
    int32_t* ord = new_order ? new_order + (int64_t)z * sel_stride + keep_indptr[r] : nullptr;
    uint32_t so = CJ_NONE, dof = CJ_NONE;
    if (B >= L) {                                        // not compacting: the order is the identity list
      const int i = chunk * 32 + lane;
      if (ord && i < L) ord[i] = sel[i];
    } else {
      const int Y = (L + P - 1) / P, X = (B + P - 1) / P;
      const int32_t start = (Y - X) * P, end = start + B;
      const int32_t p0 = start + chunk * 32, p = p0 + lane;
      int v = 0;
      if (lane == 0) v = lower_bound_i32(sel, B, start);
      if (lane == 1) v = lower_bound_i32(sel, B, end);
      if (lane == 2) v = lower_bound_i32(sel, B, p0);
      const int a = __shfl_sync(0xffffffffu, v, 0), c = __shfl_sync(0xffffffffu, v, 1), lb0 = __shfl_sync(0xffffffffu, v, 2);
      const int m = a + (B - c);                         // survivors outside the region = holes inside it
      // at most 32 kept indices fall in these 32 slots: they all sit in sel[lb0 .. lb0 + 32)
      const int wn = min(32, B - lb0);
      const int32_t win = lane < wn ? sel[lb0 + lane] : 0x7fffffff;
      const int32_t nxt = __shfl_down_sync(0xffffffffu, win, 1);
      if (lane + 1 < wn && nxt <= win) report(status, ACTKV_E_BADINDEX, r, nxt);      // must be strictly ascending
      int w = 0;                                         // #kept in [p0, p)
      bool kept = false;
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        const int32_t x = __shfl_sync(0xffffffffu, win, k);
        w += (k < wn && x < p) ? 1 : 0;
        kept = kept || (k < wn && x == p);
      }
      if (p < end) {
        if (kept) {
          if (ord) ord[p - start] = p;
        } else {
          const int j = (p - start) - (lb0 + w - a);     // rank of this hole
          if (j < 0 || j >= m) {
            report(status, ACTKV_E_BADINDEX, r, p);
          } else {
            const int32_t src_pos = j < a ? sel[j] : sel[c + (j - a)];
            if ((uint32_t)src_pos >= (uint32_t)L || (src_pos >= start && src_pos < end)) {
              report(status, ACTKV_E_BADINDEX, r, src_pos);
            } else {
              if (ord) ord[p - start] = src_pos;
              // a move whose source or destination page id is out of range is dropped (and reported)
              const int32_t sp = page_or_neg(tab, pool.n_pages, r, src_pos / P, status);
              const int32_t dp = page_or_neg(tab, pool.n_pages, r, p / P, status);
              if (sp >= 0 && dp >= 0) {
                so = (uint32_t)(((int64_t)sp * pool.stride_page + (int64_t)(src_pos % P) * pool.stride_slot +
                                 (int64_t)h * pool.stride_head) >> 3);
                dof = (uint32_t)(((int64_t)dp * pool.stride_page + (int64_t)(p % P) * pool.stride_slot +
                                  (int64_t)h * pool.stride_head) >> 3);
              }
            }
          }
        }
      }
    }
    ws->src_tab[item * 32 + lane] = so;
    ws->dst_tab[item * 32 + lane] = dof;
  }
}

// Table update: a cluster of CTAs, each with every FIN_CTAS-th request.  All of them read the old lengths (whose sums place
// the dropped pages on the free list) before any of them writes one: the cluster's barrier stands for the workspace
// that this call does not have.  6.4 us for 16 requests of 8K-24K tokens (25 when one CTA took all of them in turn).
constexpr int FIN_CTAS = 8, FIN_NT = 256;
__global__ void __cluster_dims__(FIN_CTAS, 1, 1) __launch_bounds__(FIN_NT)
    compact_inplace_finalize_kernel(TablesView tab, int32_t page_size, int32_t n_pages, const int32_t* __restrict__ budget,
                                    int32_t* status) {
  pdl_begin(budget);
  const int R = tab.n_req, tid = threadIdx.x, lane = tid & 31;
  __shared__ int64_t s_sum[FIN_NT / 32];
  const bool failed = status_set(status);
  const int32_t fc = *tab.free_count;
  auto dropped = [&](int32_t L, int32_t b) -> int32_t {      // pages that go back
    const int32_t B = b < 0 ? 0 : b;
    return B < L ? (L + page_size - 1) / page_size - (B + page_size - 1) / page_size : 0;
  };
  int64_t total = 0;
  for (int r = tid; r < R; r += FIN_NT) total += dropped(tab.seq_len[r], budget[r]);
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
  if (lane == 0) s_sum[tid >> 5] = total;
  __syncthreads();
  total = 0;
#pragma unroll
  for (int w = 0; w < FIN_NT / 32; ++w) total += s_sum[w];
  const bool ok = !failed && fc >= 0 && fc <= n_pages && fc + total <= n_pages;      // every dropped page must fit on the stack
  if (!ok && !failed && blockIdx.x == 0 && tid == 0) report(status, ACTKV_E_INVALID, -1, (int32_t)(fc + total));
  // FIN_CTAS requests at a time, one per CTA; a length is rewritten behind a barrier that every CTA reaches after it has
  // read the lengths of these requests, and the pages dropped before them are carried along.
  int64_t before = 0;
  for (int r0 = 0; r0 < R; r0 += FIN_CTAS) {
    const int q = r0 + lane;
    const bool in = lane < FIN_CTAS && q < R;
    const int32_t Lq = in ? tab.seq_len[q] : 0, bq = in ? budget[q] : 0;
    const int32_t dq = in ? dropped(Lq, bq) : 0;
    const int me = (int)blockIdx.x, r = r0 + me;
    const int64_t off = before + __reduce_add_sync(0xffffffffu, lane < me ? dq : 0);
    before += __reduce_add_sync(0xffffffffu, dq);
    const int32_t L = __shfl_sync(0xffffffffu, Lq, me), b = __shfl_sync(0xffffffffu, bq, me), drop = __shfl_sync(0xffffffffu, dq, me);
    const int32_t B = b < 0 ? 0 : b;
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (!ok || r >= R || B >= L) continue;                   // uniform over the CTA
    const int X = (B + page_size - 1) / page_size;
    int32_t* row = tab.page_table + (int64_t)r * tab.max_pages;
    for (int i = tid; i < drop; i += FIN_NT) tab.free_list[fc + off + i] = row[i];
    __syncthreads();
    // shift the row left by `drop`, chunk by chunk in ascending order: a chunk reads at or above where
    // it writes and earlier chunks wrote strictly below, so reading before the barrier is safe
    for (int i0 = 0; i0 < tab.max_pages; i0 += 4 * FIN_NT) {
      int32_t v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int i = i0 + j * FIN_NT + tid;
        v[j] = i < X ? row[i + drop] : -1;
      }
      __syncthreads();
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int i = i0 + j * FIN_NT + tid;
        if (i < tab.max_pages) row[i] = v[j];
      }
    }
    if (tid == 0) tab.seq_len[r] = B;
  }
  if (ok && blockIdx.x == 0 && tid == 0) *tab.free_count = (int32_t)(fc + total);
}

}  // namespace actkv

namespace actkv {

static int inplace_check(const actkv_pool_t* pool, const actkv_tables_t* tables, int32_t layer_begin, int32_t layer_end,
                         const int32_t* sel_idx, int64_t sel_stride, const int32_t* keep_indptr, const int32_t* budget,
                         int32_t max_keep) {
  if (!pool || !tables || !pool->base) return ACTKV_E_INVALID;
  if (layer_begin < 0 || layer_end > pool->n_layers || layer_begin > layer_end) return ACTKV_E_INVALID;
  if (pool->page_size <= 0 || pool->head_dim <= 0 || pool->head_dim % 8 != 0 || pool->n_kv_heads <= 0)
    return ACTKV_E_INVALID;
  if (((uintptr_t)pool->base & 15) || pool->stride_layer % 8 || pool->stride_kv % 8 || pool->stride_page % 8 ||
      pool->stride_slot % 8 || pool->stride_head % 8)
    return ACTKV_E_INVALID;
  const int R = tables->n_req;
  if (R < 0 || tables->max_pages < 0 || max_keep < 0 || sel_stride < 0) return ACTKV_E_INVALID;
  if (R == 0) return ACTKV_OK;
  if (!tables->page_table || !tables->seq_len || !tables->free_list || !tables->free_count || !budget ||
      !keep_indptr || !sel_idx)
    return ACTKV_E_INVALID;
  const int64_t nz = (int64_t)(layer_end - layer_begin) * pool->n_kv_heads;
  if (R > 65535 || nz > 65535) return ACTKV_E_INVALID;
  return ACTKV_OK;
}

template <int NT, int PER>
static int inplace_copy_launch(const actkv_pool_t* pool, const actkv_tables_t* tables, int32_t layer_begin, int64_t nz,
                               const int32_t* sel_idx, int64_t sel_stride, const int32_t* keep_indptr, const int32_t* budget,
                               int32_t max_keep, int32_t* new_order, int32_t* status, cudaStream_t s) {
  const PoolView pv = make_view(pool);
  const TablesView tv = make_view(tables);
  const dim3 grid((unsigned)((max_keep + NT * PER - 1) / (NT * PER)), (unsigned)tables->n_req, (unsigned)nz);
  const int vpr = pool->head_dim / 8;
  auto kern = vpr == 16  ? compact_inplace_copy_kernel<4, NT, PER>
              : vpr == 8 ? compact_inplace_copy_kernel<3, NT, PER>
              : vpr == 32 ? compact_inplace_copy_kernel<5, NT, PER>
                          : compact_inplace_copy_kernel<-1, NT, PER>;
  // (launched plainly: with its CTAs placed while the selection kernel drains, the 16-request copy takes 571 us, not 455;
  //  they then seem to keep that kernel's division of the SM between shared memory and L1)
  kern<<<grid, NT, 0, s>>>(pv, tv, layer_begin, sel_idx, sel_stride, keep_indptr, budget, max_keep, new_order, status);
  ACTKV_CHECK_LAUNCH();
  return ACTKV_OK;
}

// The whole copy of a call in one launch.
static int inplace_copy_all(const actkv_pool_t* pool, const actkv_tables_t* tables, int32_t layer_begin, int32_t layer_end,
                            const int32_t* sel_idx, int64_t sel_stride, const int32_t* keep_indptr, const int32_t* budget,
                            int32_t max_keep, int32_t* new_order, int32_t* status, cudaStream_t s) {
  const int64_t nz = (int64_t)(layer_end - layer_begin) * pool->n_kv_heads;
  if (nz <= 0 || max_keep <= 0) return ACTKV_OK;
  // 256 slots per CTA, 128 while that would leave fewer than four CTAs per SM.  (512 slots: 454 us where 256 take 463 at
  // 80 % kept, but 486 for 478 at 25 % and 99 for 93 at one layer.)
  if (((int64_t)max_keep + 255) / 256 * tables->n_req * nz >= 4 * 148)
    return inplace_copy_launch<128, 2>(pool, tables, layer_begin, nz, sel_idx, sel_stride, keep_indptr, budget, max_keep,
                                       new_order, status, s);
  return inplace_copy_launch<128, 1>(pool, tables, layer_begin, nz, sel_idx, sel_stride, keep_indptr, budget, max_keep, new_order,
                                     status, s);
}

static int inplace_finalize(const actkv_pool_t* pool, const actkv_tables_t* tables, int32_t layer_end, const int32_t* budget,
                            int32_t* status, cudaStream_t s) {
  if (layer_end == pool->n_layers) {
    launch_pdl(compact_inplace_finalize_kernel, FIN_CTAS, FIN_NT, 0, s, make_view(tables),
               pool->page_size, pool->n_pages, budget, status);
    ACTKV_CHECK_LAUNCH();
  }
  return ACTKV_OK;
}

// Items of the largest job these arguments allow, per layer.
static int64_t inplace_items_per_layer(const actkv_pool_t* pool, int32_t n_req, int32_t max_keep) {
  return (int64_t)pool->n_kv_heads * n_req * (((int64_t)max_keep + 31) / 32);
}
static size_t inplace_ws_base(int32_t n_req) {
  return align_up(sizeof(CompactWs) + sizeof(int32_t) * ((size_t)3 * n_req + 1), 256);
}

}  // namespace actkv

extern "C" {

int actkv_compact_inplace(const actkv_pool_t* pool, const actkv_tables_t* tables, int32_t layer_begin,
                          int32_t layer_end, const int32_t* sel_idx, int64_t sel_stride,
                          const int32_t* keep_indptr, const int32_t* budget, int32_t max_keep,
                          int32_t* new_order, int32_t* status, actkv_stream_t stream) {
  using namespace actkv;
  int rc = inplace_check(pool, tables, layer_begin, layer_end, sel_idx, sel_stride, keep_indptr, budget, max_keep);
  if (rc != ACTKV_OK || tables->n_req == 0) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  rc = inplace_copy_all(pool, tables, layer_begin, layer_end, sel_idx, sel_stride, keep_indptr, budget, max_keep, new_order,
                        status, s);
  if (rc != ACTKV_OK) return rc;
  return inplace_finalize(pool, tables, layer_end, budget, status, s);
}

size_t actkv_compact_inplace_deferred_workspace_bytes(const actkv_pool_t* pool, int32_t n_req, int32_t n_layers_sub,
                                                      int32_t max_keep) {
  if (!pool || n_req < 0 || n_layers_sub < 0 || max_keep < 0 || pool->n_kv_heads <= 0) return 0;
  const int64_t items = actkv::inplace_items_per_layer(pool, n_req, max_keep) * n_layers_sub;
  return actkv::inplace_ws_base(n_req) + 2 * actkv::align_up((size_t)items * 32 * sizeof(uint32_t), 256);
}

int actkv_compact_inplace_begin(const actkv_pool_t* pool, const actkv_tables_t* tables, int32_t layer_begin,
                                int32_t layer_end, const int32_t* sel_idx, int64_t sel_stride,
                                const int32_t* keep_indptr, const int32_t* budget, int32_t max_keep,
                                int32_t* new_order, void* ws, size_t ws_bytes, int32_t* status, actkv_stream_t stream) {
  using namespace actkv;
  int rc = inplace_check(pool, tables, layer_begin, layer_end, sel_idx, sel_stride, keep_indptr, budget, max_keep);
  if (rc != ACTKV_OK || tables->n_req == 0) return rc;
  if (!ws || ws_bytes < inplace_ws_base(tables->n_req)) return ACTKV_E_WORKSPACE;
  cudaStream_t s = (cudaStream_t)stream;
  const int nl = layer_end - layer_begin;
  const int shift = deferrable_shift(pool);
  const int64_t items_max = inplace_items_per_layer(pool, tables->n_req, max_keep) * nl;
  const bool deferred = shift >= 0 && items_max <= 0x7fffffff &&
                        ws_bytes >= actkv_compact_inplace_deferred_workspace_bytes(pool, tables->n_req, nl, max_keep);
  const size_t base = inplace_ws_base(tables->n_req);
  const size_t tab_bytes = align_up((size_t)(deferred ? items_max : 0) * 32 * sizeof(uint32_t), 256);
  uint32_t* src_tab = (uint32_t*)((char*)ws + base);
  uint32_t* dst_tab = (uint32_t*)((char*)ws + base + tab_bytes);
  // (not deferred: an empty job, so that a score call given this workspace finds nothing to do; actkv_compact_inplace_end
  //  then copies everything itself)
  launch_pdl(compact_inplace_plan_kernel, 1, 32, 0, s, make_view(tables), make_view(pool), budget, max_keep,
             new_order != nullptr ? 1 : 0, layer_begin, deferred ? nl : 0, deferred ? shift : -1, src_tab, dst_tab,
             deferred ? items_max : 0, (CompactWs*)ws, status);
  ACTKV_CHECK_LAUNCH();
  if (deferred && items_max > 0) {
    const int64_t ctas = std::min<int64_t>(std::max<int64_t>(1, (items_max + 3) / 4), 1 << 20);
    launch_pdl(compact_inplace_resolve_kernel, (unsigned)ctas, 128, 0, s, (CompactWs*)ws, sel_idx, sel_stride, keep_indptr,
               new_order);
    ACTKV_CHECK_LAUNCH();
  }
  return ACTKV_OK;
}

int actkv_compact_inplace_end(const actkv_pool_t* pool, const actkv_tables_t* tables, int32_t layer_begin,
                              int32_t layer_end, const int32_t* sel_idx, int64_t sel_stride,
                              const int32_t* keep_indptr, const int32_t* budget, int32_t max_keep,
                              int32_t* new_order, void* ws, size_t ws_bytes, int32_t* status, actkv_stream_t stream) {
  using namespace actkv;
  int rc = inplace_check(pool, tables, layer_begin, layer_end, sel_idx, sel_stride, keep_indptr, budget, max_keep);
  if (rc != ACTKV_OK || tables->n_req == 0) return rc;
  if (!ws || ws_bytes < inplace_ws_base(tables->n_req)) return ACTKV_E_WORKSPACE;
  cudaStream_t s = (cudaStream_t)stream;
  const int nl = layer_end - layer_begin;
  const int shift = deferrable_shift(pool);
  const int64_t items_max = inplace_items_per_layer(pool, tables->n_req, max_keep) * nl;
  const bool deferred = shift >= 0 && items_max <= 0x7fffffff &&
                        ws_bytes >= actkv_compact_inplace_deferred_workspace_bytes(pool, tables->n_req, nl, max_keep);
  if (!deferred) {
    rc = inplace_copy_all(pool, tables, layer_begin, layer_end, sel_idx, sel_stride, keep_indptr, budget, max_keep, new_order,
                          status, s);
    if (rc != ACTKV_OK) return rc;
  } else if (items_max > 0) {
    launch_drain((CompactWs*)ws, shift, items_max, s);
    ACTKV_CHECK_LAUNCH();
  }
  return inplace_finalize(pool, tables, layer_end, budget, status, s);
}

}  // extern "C"
