// Warp-level tensor-core path of actkv_score (mma.sync m16n8k16, bf16 in, fp32 accumulate): short windows (fewer than
// 64 window x group rows, where a 128-row tcgen05 tile would be mostly padding) and every pool layout the tcgen05
// kernels do not take: any head_dim (multiple of 8, <= 256), any page size and strides, any window.
//
// Section 7.1 / Algorithm 3: s = q.k, A = exp(s - LSE), max over the GQA group, mean over the action tokens.  Logits
// are kept in log2 units (t = s * sm_scale * log2 e) so that exp2 maps to one MUFU op.
//
// What bounds it: the K reads.  At 32 rows a key costs 8 KFLOP against 256 bytes, so both passes should run at the
// HBM rate; with fp32 FMAs (the kernel this one replaced) they were bound by arithmetic and shared-memory loads:
// 5.05 and 4.57 ms for 7.4 M (key, head, layer) rows of 128 dims against 12-48 window rows.
// Here: 0.39 and 0.44 ms (4.8 and 4.3 TB/s of K reads); what is left of the distance to 6.5 TB/s is the issue rate of
// the matrix instructions (one m16n8k16 per 8.5 cycles and scheduler) and of the folds between them.  Long windows on
// layouts of this path are bound by that rate: 256 rows at head_dim 96 4.37 and 3.34 -> 0.47 and 0.47 ms, 512 rows at
// pages of 8 tokens 5.52 and 4.16 -> 0.48 and 0.52 ms (188 and 173 TFLOP/s).
// Loads go through a ring in shared memory and not to registers ahead of time: the registers are what limits the
// resident warps (four CTAs of 128 threads; with two and twice the ring 0.45 and 0.52 ms).
//
// Layout.  The order of the head dimensions is the same on both sides of a product and otherwise free, so a thread's
// fragments are whole 16-byte vectors: lane l holds dims 32 b + 8 (l % 4) .. + 7 of key l / 4 and of row l / 4;
// elements 0-3 of a vector are one k16 step and elements 4-7 the next.  The pooled-score pass computes D[key, row]
// (max over the group and sum over the tokens need at most two shuffles), the LSE pass D[row, key] (a thread owns two
// rows of a tile and folds their logits without any).  A warp takes 32 keys at a time (16 at head_dim > 128) from a
// ring of its own and keeps them in registers for all rows of a chunk.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace actkv {

constexpr int MAX_GROUP = 32;     // query heads per KV head
constexpr int LSE_CHUNK = 512;    // fewest keys per partial (m, sum) of the LSE pass (both paths)
constexpr int LSE_CHUNK_LONG = 4096;  // fewest keys per partial while the launch still has LSE_ITEMS_MIN work items
constexpr int LSE_ITEMS = 20 * 148;  // work items an LSE launch aims for: 20 per SM
constexpr int LSE_ITEMS_MIN = 4 * 148;

struct ScoreArgs {
  PoolView pool;
  TablesView tab;
  const __nv_bfloat16* q;        // [NLs, sum_win, Hq, D]
  const int32_t* win_indptr;
  const int32_t* tok_indptr;
  const float* lse;              // [NLs, sum_win, Hq] natural log (pass 2 input)
  float2* partials;              // [units, n_chunks, rows_max] (pass 1 output), log2 units
  float* score_out;              // [NLs, Hkv, sum_tok]
  int32_t* status;
  int32_t layer_begin, n_layers_sub, n_q_heads, group;
  int32_t sum_win, sum_tok, rows_max, n_chunks;
  int32_t lse_chunk;             // keys per LSE partial of this launch (multiple of 128, >= LSE_CHUNK)
  int32_t page_shift;            // log2(page_size), -1 when it is not a power of two
  float scale_log2;              // sm_scale * log2(e)
  int32_t causal;
  int32_t win_left;              // sliding-window layer: a query at position p sees keys p - win_left < j <= p (0: all)
  const int32_t* acc_steps;      // accumulate mode (streaming, Algorithm 3 step 5): [R] action queries already
                                 // folded into score_out; nullptr: score_out is overwritten with this call's mean
};

// What is stored for one key: the mean over this call's W action tokens (`mean_w`), or in accumulate
// mode the running mean over the n earlier action tokens of the region and this call's W
// (n = 0: the old value is not read, the state restarts).
__device__ __forceinline__ void store_pooled(const ScoreArgs& a, int r, float* slot, float sum_w, float mean_w, int W) {
  if (a.acc_steps != nullptr) {
    const int n = a.acc_steps[r];
    if (n > 0) mean_w = fmaf(*slot, (float)n, sum_w) / (float)(n + W);
  }
  *slot = mean_w;
}

namespace wm {

constexpr int NT = 128;           // threads per CTA: four warps
constexpr int WARPS = NT / 32;
constexpr int RCH = 64;           // rows per chunk (the keys are read again for every further chunk)
constexpr float NO_REF = -3.402823466e38f;     // LSE pass: the reference before the first visible logit (finite: its sum is 0)
constexpr int POOL_KEYS = 2048;   // keys per CTA of the pooled-score pass (at most; 1024 and 4096 measured 1-3 % slower)

__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t bytes) {     // the rest of 16 is zeroed
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// DB: 32-dim blocks of the head dimension (dims past head_dim are zeros on both sides).
template <int DB>
struct Keys {
  static constexpr int MT = DB > 4 ? 1 : 2;       // 16-key tiles
  static constexpr int N = 16 * MT;               // keys a warp holds
  static constexpr int VECS = MT * 2 * DB;        // 16-byte vectors per lane
  static constexpr int STAGES = 16 / VECS;        // tiles of a warp's ring: 8 KB in flight, four warps, four CTAs per SM
  uint4 v[MT][2][DB];                             // [tile][key l/4 or l/4 + 8][block]
};
template <int DB>
struct Smem {
  uint4 ring[WARPS][Keys<DB>::STAGES][Keys<DB>::VECS][32];
  uint4 sq[RCH / 8 * DB * 32];
  union {
    float nlse[RCH];                              // pooled-score pass
    float2 red[WARPS * RCH];                      // LSE pass: the warps' (reference, sum)
  };
};

// Element offset of key `key` of request r within its layer and head, -1 past the end of the request.
__device__ __forceinline__ int64_t key_offset(const ScoreArgs& a, int r, int key, int L) {
  if (key >= L) return -1;
  const int P = a.pool.page_size;
  const int lp = a.page_shift >= 0 ? key >> a.page_shift : key / P;
  const int page = checked_page(a.tab, a.pool.n_pages, r, lp, a.status);
  return (int64_t)page * a.pool.stride_page + (int64_t)(key - lp * P) * a.pool.stride_slot;
}

// A warp's K tiles key0, key0 + step, ... below key_end through its ring.  Every lane copies exactly the vectors it will
// itself hold (cp.async into slots in lane order: no bank conflicts, no synchronisation beyond the lane's own wait).
template <int DB>
struct KeyStream {
  using K = Keys<DB>;
  const ScoreArgs& a;
  const __nv_bfloat16* kbase;
  uint32_t ring;               // shared address of this lane's first slot
  int r, L, D, lane, step, key_end, next, stage;
  int64_t off;                 // key_offset of key (lane % N) of tile `next`
  __device__ __forceinline__ KeyStream(const ScoreArgs& a_, const __nv_bfloat16* kb, uint4* ring_, int r_, int L_, int lane_,
                                       int key0, int step_, int end)
      : a(a_), kbase(kb), ring((uint32_t)__cvta_generic_to_shared(ring_ + lane_)), r(r_), L(L_), D(a_.pool.head_dim), lane(lane_),
        step(step_), key_end(end), next(key0), stage(0) {
    off = next < key_end ? key_offset(a, r, next + lane % K::N, L) : -1;
#pragma unroll
    for (int i = 0; i < K::STAGES; ++i) issue(i);
  }
  __device__ __forceinline__ void issue(int s) {
    if (next < key_end) {      // (uniform over the warp)
      const int t = lane & 3;
      const bool plain = next + K::N <= L && D == DB * 32;       // nothing to zero
#pragma unroll
      for (int i = 0; i < 2 * K::MT; ++i) {
        const int64_t o = __shfl_sync(0xffffffffu, off, i * 8 + (lane >> 2));
        const uint32_t dst = ring + (s * K::VECS + i * DB) * 512;
        const __nv_bfloat16* src = kbase + (plain || o >= 0 ? o : 0) + t * 8;
        if (plain) {
#pragma unroll
          for (int b = 0; b < DB; ++b) cp_async16(dst + b * 512, src + b * 32, 16u);
        } else {
#pragma unroll
          for (int b = 0; b < DB; ++b) {
            const bool live = o >= 0 && (b * 4 + t) * 8 < D;
            cp_async16(dst + b * 512, live ? src + b * 32 : kbase, live ? 16u : 0u);
          }
        }
      }
      next += step;
      off = next < key_end ? key_offset(a, r, next + lane % K::N, L) : -1;
    }
    cp_commit();
  }
  // the next tile into registers; its slots are refilled at once
  __device__ __forceinline__ void take(K& k) {
    cp_wait<K::STAGES - 1>();
#pragma unroll
    for (int i = 0; i < 2 * K::MT; ++i)
#pragma unroll
      for (int b = 0; b < DB; ++b) {
        uint4& v = k.v[i >> 1][i & 1][b];
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                     : "r"(ring + (stage * K::VECS + i * DB + b) * 512) : "memory");
      }
    __syncwarp();              // the slots have been read before they are written again
    issue(stage);
    if (++stage == K::STAGES) stage = 0;
  }
};

// acc[q][mt] = K Q^T of n-tiles nt0 .. nt0 + NG - 1
template <int DB, int NG>
__device__ __forceinline__ void contract(float (&acc)[NG][Keys<DB>::MT][4], const Keys<DB>& k, const uint4* sq, int nt0, int lane) {
#pragma unroll
  for (int q = 0; q < NG; ++q)
#pragma unroll
    for (int mt = 0; mt < Keys<DB>::MT; ++mt)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[q][mt][i] = 0.f;
#pragma unroll
  for (int b = 0; b < DB; ++b)
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      const uint4 w = sq[((nt0 + q) * DB + b) * 32 + lane];
#pragma unroll
      for (int mt = 0; mt < Keys<DB>::MT; ++mt) {
        mma16816(acc[q][mt], k.v[mt][0][b].x, k.v[mt][1][b].x, k.v[mt][0][b].y, k.v[mt][1][b].y, w.x, w.y);
        mma16816(acc[q][mt], k.v[mt][0][b].z, k.v[mt][1][b].z, k.v[mt][0][b].w, k.v[mt][1][b].w, w.z, w.w);
      }
    }
}

// Rows [row0, row0 + 8 n_nt) of the unit, row = w * gp + g, into shared memory in lane order; zeros for rows past the
// window, padding heads (g >= G) and dims past head_dim.  `flip`: the sign bits of a pair (0x80008000 negates the rows).
template <int DB>
__device__ __forceinline__ void load_rows(uint4* sq, const __nv_bfloat16* qbase, int row0, int n_nt, int W, int gp, int G,
                                          int n_q_heads, int D, uint32_t flip = 0u) {
  for (int i = threadIdx.x; i < n_nt * DB * 32; i += NT) {
    const int l = i & 31, b = (i >> 5) % DB, nt = (i >> 5) / DB;
    const int n = row0 + nt * 8 + (l >> 2), w = n / gp, g = n - w * gp, d = (b * 4 + (l & 3)) * 8;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (w < W && g < G && d < D) v = __ldg(reinterpret_cast<const uint4*>(qbase + ((int64_t)w * n_q_heads + g) * D + d));
    sq[i] = make_uint4(v.x ^ flip, v.y ^ flip, v.z ^ flip, v.w ^ flip);
  }
}

// What both passes need to know about their unit.
struct Unit {
  int r, h, slab, L, w0, W;
  const __nv_bfloat16 *kbase, *qbase;
};
__device__ __forceinline__ Unit unit_of(const ScoreArgs& a, int u) {
  Unit x;
  const int R = a.tab.n_req, Hkv = a.pool.n_kv_heads;
  x.r = u % R;
  x.h = (u / R) % Hkv;
  x.slab = u / (R * Hkv);
  x.L = a.tab.seq_len[x.r];
  x.w0 = a.win_indptr[x.r];
  x.W = a.win_indptr[x.r + 1] - x.w0;
  x.kbase = a.pool.base + (int64_t)(a.layer_begin + x.slab) * a.pool.stride_layer + (int64_t)x.h * a.pool.stride_head;
  x.qbase = a.q + (((int64_t)x.slab * a.sum_win + x.w0) * a.n_q_heads + (int64_t)x.h * a.group) * a.pool.head_dim;
  return x;
}

// LSE pass: partial (reference, sum of exp2) of every window row over one chunk of lse_chunk keys.
template <int DB>
__global__ void __launch_bounds__(NT, 4) score_mma_lse_kernel(const ScoreArgs a) {
  pdl_begin();
  constexpr int KN = Keys<DB>::N, NK = KN / 8, MTILES = RCH / 16;
  extern __shared__ __align__(16) uint8_t wm_smem[];
  Smem<DB>& sm = *reinterpret_cast<Smem<DB>*>(wm_smem);
  uint4* sq = sm.sq;
  float2* red = sm.red;
  const int u = blockIdx.x / a.n_chunks, chunk = blockIdx.x - u * a.n_chunks;
  const Unit x = unit_of(a, u);
  const int L = x.L, W = x.W, G = a.group, D = a.pool.head_dim;
  const int key_begin = chunk * a.lse_chunk;
  if (key_begin >= L) return;
  if (W <= 0 || (a.causal && W > L)) {               // no window, or a window longer than the cache
    if (threadIdx.x == 0 && chunk == 0) report(a.status, ACTKV_E_INVALID, x.r, W);
    return;
  }
  const int rows = W * G;
  if (rows > a.rows_max || L > a.n_chunks * a.lse_chunk) {      // the host sized the partials from upper bounds
    if (threadIdx.x == 0 && chunk == 0) report(a.status, ACTKV_E_INVALID, x.r, rows > a.rows_max ? W : L);
    return;
  }
  const int key_end = min(L, key_begin + a.lse_chunk);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t = lane & 3;
  // keys below lo_all are seen by no row (sliding-window layer), keys in [lo_every, hi_every] by every row
  const int p_first = a.causal ? L - W : L - 1, p_last = L - 1;
  const int lo_all = a.win_left > 0 ? max(0, p_first - a.win_left + 1) : 0;
  const int lo_every = a.win_left > 0 ? max(0, p_last - a.win_left + 1) : 0, hi_every = p_first;
  const int key_first = max(key_begin, lo_all / KN * KN) + warp * KN;
  // (a negative scale is taken into the rows, so that the maxima are maxima of the scaled logits)
  const float c = fmaxf(fabsf(a.scale_log2), 1e-35f);
  const uint32_t flip = a.scale_log2 < 0.f ? 0x80008000u : 0u;

  for (int row0 = 0; row0 < rows; row0 += RCH) {
    const int n_mt = (min(rows - row0, RCH) + 15) / 16;
    __syncthreads();
    KeyStream<DB> ks(a, x.kbase, &sm.ring[warp][0][0][0], x.r, L, lane, key_first, WARPS * KN, key_end);
    load_rows<DB>(sq, x.qbase, row0, 2 * n_mt, W, G, G, a.n_q_heads, D, flip);
    __syncthreads();
    float m[MTILES][2], s[MTILES][2];                // of rows 16 p + 8 i + l / 4
#pragma unroll
    for (int p = 0; p < MTILES; ++p)
#pragma unroll
      for (int i = 0; i < 2; ++i) { m[p][i] = NO_REF; s[p][i] = 0.f; }
    for (int key0 = key_first; key0 < key_end; key0 += WARPS * KN) {
      Keys<DB> k;
      ks.take(k);
      const bool whole = key0 >= lo_every && key0 + KN - 1 <= hi_every;
#pragma unroll
      for (int p = 0; p < MTILES; ++p) {
        if (p >= n_mt) continue;
        float acc[NK][4];
#pragma unroll
        for (int j = 0; j < NK; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
#pragma unroll
        for (int b = 0; b < DB; ++b) {
          const uint4 q0 = sq[((2 * p) * DB + b) * 32 + lane], q1 = sq[((2 * p + 1) * DB + b) * 32 + lane];
#pragma unroll
          for (int j = 0; j < NK; ++j) mma16816(acc[j], q0.x, q1.x, q0.y, q1.y, k.v[j >> 1][j & 1][b].x, k.v[j >> 1][j & 1][b].y);
#pragma unroll
          for (int j = 0; j < NK; ++j) mma16816(acc[j], q0.z, q1.z, q0.w, q1.w, k.v[j >> 1][j & 1][b].z, k.v[j >> 1][j & 1][b].w);
        }
        if (!whole) {
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int w = min((row0 + 16 * p + 8 * i + (lane >> 2)) / G, W - 1);
            const int last = a.causal ? L - W + w : L - 1;
#pragma unroll
            for (int j = 0; j < 2 * NK; ++j) {
              const int key = key0 + (j >> 1) * 8 + 2 * t + (j & 1);
              if (key > last || (a.win_left > 0 && key <= last - a.win_left)) acc[j >> 1][2 * i + (j & 1)] = -INFINITY;
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          float mx = fmaxf(acc[0][2 * i], acc[0][2 * i + 1]);
#pragma unroll
          for (int j = 1; j < NK; ++j) mx = fmaxf(mx, fmaxf(acc[j][2 * i], acc[j][2 * i + 1]));
          mx = __fmul_ru(mx, c);   // (rounded up: of a huge maximum the exponent below is then at most 0)
          // the reference follows the maximum only when it has fallen behind by 2^16: the sum stays far below overflow
          if (mx > m[p][i] + 16.f) { s[p][i] *= exp2f(m[p][i] - mx); m[p][i] = mx; }
          float e = 0.f;
#pragma unroll
          for (int j = 0; j < 2 * NK; ++j) e += exp2f(fmaf(acc[j >> 1][2 * i + (j & 1)], c, -m[p][i]));
          s[p][i] += e;
        }
      }
    }
    // over the four lanes of a row, then over the warps
#pragma unroll
    for (int p = 0; p < MTILES; ++p) {
      if (p >= n_mt) continue;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) {
          const float m2 = __shfl_xor_sync(0xffffffffu, m[p][i], o), s2 = __shfl_xor_sync(0xffffffffu, s[p][i], o);
          const float mm = fmaxf(m[p][i], m2);
          s[p][i] = s[p][i] * exp2f(m[p][i] - mm) + s2 * exp2f(m2 - mm);
          m[p][i] = mm;
        }
        if (t == 0) red[warp * RCH + 16 * p + 8 * i + (lane >> 2)] = make_float2(m[p][i], s[p][i]);
      }
    }
    __syncthreads();
    for (int n = threadIdx.x; n < min(rows - row0, RCH); n += NT) {
      float mm = red[n].x;
#pragma unroll
      for (int w = 1; w < WARPS; ++w) mm = fmaxf(mm, red[w * RCH + n].x);
      float ss = 0.f;
#pragma unroll
      for (int w = 0; w < WARPS; ++w) ss += red[w * RCH + n].y * exp2f(red[w * RCH + n].x - mm);
      // a row that sees none of these keys has no reference; a sum of 0 beside one is that of logits whose rounding alone is
      // beyond the range of exp2 (the largest counts 1); a NaN is handed on
      a.partials[((int64_t)u * a.n_chunks + chunk) * a.rows_max + row0 + n] =
          mm == NO_REF && ss == 0.f ? make_float2(-INFINITY, 0.f) : make_float2(mm, ss == 0.f ? 1.f : ss);
    }
  }
}

// Pooled-score pass: the scores of keys_per_cta keys.  GP: the group size rounded up to a power of two; the padding
// heads drop out of the max (-lse = -inf).
template <int DB, int GP>
__global__ void __launch_bounds__(NT, 4) score_mma_pool_kernel(const ScoreArgs a, int keys_per_cta, int n_parts) {
  pdl_begin();
  constexpr int MT = Keys<DB>::MT, KN = Keys<DB>::N, NG = GP == 32 ? 4 : 2;
  extern __shared__ __align__(16) uint8_t wm_smem[];
  Smem<DB>& sm = *reinterpret_cast<Smem<DB>*>(wm_smem);
  uint4* sq = sm.sq;
  float* nlse = sm.nlse;
  const int u = blockIdx.x / n_parts, part = blockIdx.x - u * n_parts;
  const Unit x = unit_of(a, u);
  const int L = x.L, W = x.W, G = a.group, D = a.pool.head_dim;
  const int key_begin = part * keys_per_cta;
  if (key_begin >= L) return;
  if (W <= 0 && a.acc_steps != nullptr) return;      // accumulate mode: a request outside its action region
  if (W <= 0 || (a.causal && W > L)) {
    if (threadIdx.x == 0 && part == 0) report(a.status, ACTKV_E_INVALID, x.r, W);
    return;
  }
  if (L > n_parts * keys_per_cta) {
    if (threadIdx.x == 0 && part == 0) report(a.status, ACTKV_E_INVALID, x.r, L);
    return;
  }
  const int key_end = min(L, key_begin + keys_per_cta);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t = lane & 3;
  const int win = a.win_left, lw = L - W;
  const int p_first = a.causal ? lw : L - 1, p_last = L - 1;
  const int lo_all = win > 0 ? max(0, p_first - win + 1) : 0;
  const int lo_every = win > 0 ? max(0, p_last - win + 1) : 0, hi_every = p_first;
  const int key_first = max(key_begin, lo_all / KN * KN) + warp * KN;
  const float c = a.scale_log2;
  const float* lse_base = a.lse + ((int64_t)x.slab * a.sum_win + x.w0) * a.n_q_heads + x.h * G;
  float* out = a.score_out + ((int64_t)x.slab * a.pool.n_kv_heads + x.h) * a.sum_tok + a.tok_indptr[x.r];
  // the first chunk of rows forms the mean (with the n already folded in: (n Out + S) / (n + W)), later ones add S / (n + W)
  const float inv_w = 1.f / (float)(W + (a.acc_steps != nullptr ? a.acc_steps[x.r] : 0));
  for (int key = key_begin + threadIdx.x; key < min(key_end, lo_all / KN * KN); key += NT)      // seen by no row
    store_pooled(a, x.r, out + key, 0.f, 0.f, W);

  for (int row0 = 0; row0 < W * GP; row0 += RCH) {
    const int n_nt = (min(W * GP - row0, RCH) + 8 * NG - 1) / (8 * NG) * NG;
    __syncthreads();
    KeyStream<DB> ks(a, x.kbase, &sm.ring[warp][0][0][0], x.r, L, lane, key_first, WARPS * KN, key_end);
    load_rows<DB>(sq, x.qbase, row0, n_nt, W, GP, G, a.n_q_heads, D);
    for (int n = threadIdx.x; n < n_nt * 8; n += NT) {
      const int w = (row0 + n) / GP, g = (row0 + n) % GP;
      nlse[n] = (w < W && g < G) ? -lse_base[(int64_t)w * a.n_q_heads + g] * kLog2e : -INFINITY;
    }
    __syncthreads();
    for (int key0 = key_first; key0 < key_end; key0 += WARPS * KN) {
      Keys<DB> k;
      ks.take(k);
      const bool whole = key0 >= lo_every && key0 + KN - 1 <= hi_every;
      float sum[MT][2];
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) sum[mt][0] = sum[mt][1] = 0.f;
      for (int nt = 0; nt < n_nt; nt += NG) {
        float acc[NG][MT][4];
        contract<DB, NG>(acc, k, sq, nt, lane);
        // (s c - lse) of this thread's two columns of every n-tile
#pragma unroll
        for (int q = 0; q < NG; ++q) {
          const float2 nl = *reinterpret_cast<const float2*>(&nlse[(nt + q) * 8 + 2 * t]);
#pragma unroll
          for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              acc[q][mt][2 * h] = fmaf(acc[q][mt][2 * h], c, nl.x);
              acc[q][mt][2 * h + 1] = fmaf(acc[q][mt][2 * h + 1], c, nl.y);
            }
        }
        // max over the group, exp, sum over the tokens: a token's GP columns lie in one thread (GP <= 2), in 2 or 4
        // lanes (4, 8) or in 4 lanes of GP / 8 n-tiles (16, 32); all of its lanes then hold the same sum
        constexpr int QG = GP > 8 ? GP / 8 : 1;      // n-tiles per token
        auto fold = [&](auto all) {
#pragma unroll
          for (int q = 0; q < NG; q += QG)
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                auto add = [&](float y, int n) {
                  float e = fmaxf(exp2f(y), 0.f);    // (NaN, as padding rows give with an infinite key, counts as nothing)
                  if constexpr (!decltype(all)::value) {
                    const int key = key0 + mt * 16 + h * 8 + (lane >> 2), w = n / GP;
                    const int w_min = a.causal ? max(0, key - lw) : 0;
                    const int w_end = win > 0 ? (a.causal ? min(W, key - lw + win) : (key >= L - win ? W : 0)) : W;
                    if (w < w_min || w >= w_end) e = 0.f;
                  }
                  sum[mt][h] += e;
                };
                const int n = row0 + (nt + q) * 8 + 2 * t;
                if constexpr (GP == 1) {
                  add(acc[q][mt][2 * h], n);
                  add(acc[q][mt][2 * h + 1], n + 1);
                } else {
                  float mx = fmaxf(acc[q][mt][2 * h], acc[q][mt][2 * h + 1]);
#pragma unroll
                  for (int j = 1; j < QG; ++j) mx = fmaxf(mx, fmaxf(acc[q + j][mt][2 * h], acc[q + j][mt][2 * h + 1]));
                  if (GP >= 4) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                  if (GP >= 8) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
                  add(mx, n);
                }
              }
        };
        if (whole) fold(std::true_type{}); else fold(std::false_type{});
      }
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float y = sum[mt][h];
          if (GP <= 2) y += __shfl_xor_sync(0xffffffffu, y, 1);
          if (GP <= 4) y += __shfl_xor_sync(0xffffffffu, y, 2);
          const int key = key0 + mt * 16 + h * 8 + (lane >> 2);
          if (t == 0 && key < key_end) {
            if (row0 == 0) store_pooled(a, x.r, out + key, y, y * inv_w, W);
            else out[key] += y * inv_w;
          }
        }
    }
  }
}

template <int DB>
inline int launch_lse_d(const ScoreArgs& a, unsigned grid, cudaStream_t s) {
  if (ensure_dyn_smem(score_mma_lse_kernel<DB>, sizeof(Smem<DB>)) != cudaSuccess) return ACTKV_E_CUDA;
  launch_pdl(score_mma_lse_kernel<DB>, grid, NT, sizeof(Smem<DB>), s, a);
  ACTKV_CHECK_LAUNCH();
  return ACTKV_OK;
}

inline int launch_lse(const ScoreArgs& a, int64_t units, cudaStream_t s) {
  const int64_t grid = units * a.n_chunks;
  if (grid > 0x7fffffffLL) return ACTKV_E_INVALID;
  if (a.pool.head_dim <= 64) return launch_lse_d<2>(a, (unsigned)grid, s);
  if (a.pool.head_dim <= 128) return launch_lse_d<4>(a, (unsigned)grid, s);
  return launch_lse_d<8>(a, (unsigned)grid, s);
}

template <int DB, int GP>
inline int launch_pool_g(const ScoreArgs& a, unsigned grid, int keys, int parts, cudaStream_t s) {
  if (ensure_dyn_smem(score_mma_pool_kernel<DB, GP>, sizeof(Smem<DB>)) != cudaSuccess) return ACTKV_E_CUDA;
  launch_pdl(score_mma_pool_kernel<DB, GP>, grid, NT, sizeof(Smem<DB>), s, a, keys, parts);
  ACTKV_CHECK_LAUNCH();
  return ACTKV_OK;
}

template <int DB>
inline int launch_pool_d(const ScoreArgs& a, unsigned grid, int keys, int parts, cudaStream_t s) {
  if (a.group <= 1) return launch_pool_g<DB, 1>(a, grid, keys, parts, s);
  if (a.group <= 2) return launch_pool_g<DB, 2>(a, grid, keys, parts, s);
  if (a.group <= 4) return launch_pool_g<DB, 4>(a, grid, keys, parts, s);
  if (a.group <= 8) return launch_pool_g<DB, 8>(a, grid, keys, parts, s);
  if (a.group <= 16) return launch_pool_g<DB, 16>(a, grid, keys, parts, s);
  return launch_pool_g<DB, 32>(a, grid, keys, parts, s);
}

inline int launch_pool(const ScoreArgs& a, int64_t units, int max_tok, cudaStream_t s) {
  // as many keys per CTA as leave 16 CTAs per SM (four rounds of four resident ones): a CTA loads its rows and fills
  // its rings first
  int keys = POOL_KEYS;
  while (keys > 128 && units * ((max_tok + keys - 1) / keys) < 16 * 148) keys >>= 1;
  const int parts = (max_tok + keys - 1) / keys;
  const int64_t grid = units * parts;
  if (grid > 0x7fffffffLL) return ACTKV_E_INVALID;
  if (a.pool.head_dim <= 64) return launch_pool_d<2>(a, (unsigned)grid, keys, parts, s);
  if (a.pool.head_dim <= 128) return launch_pool_d<4>(a, (unsigned)grid, keys, parts, s);
  return launch_pool_d<8>(a, (unsigned)grid, keys, parts, s);
}

}  // namespace wm

// Merges the per-chunk (max, sum) partials of one window row into its LSE (natural log units).
__global__ void lse_combine_kernel(const ScoreArgs a, float* lse_out) {
  pdl_begin();
  const int R = a.tab.n_req, Hkv = a.pool.n_kv_heads, G = a.group;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;   // over units * rows_max
  const int64_t total = (int64_t)a.n_layers_sub * Hkv * R * a.rows_max;
  if (idx >= total) return;
  const int row = (int)(idx % a.rows_max);
  const int u = (int)(idx / a.rows_max);
  const int r = u % R, h = (u / R) % Hkv, slab = u / (R * Hkv);
  const int L = a.tab.seq_len[r];
  const int w0 = a.win_indptr[r], W = a.win_indptr[r + 1] - w0;
  if (row >= W * G || L <= 0) return;
  const int n_chunks = (L + a.lse_chunk - 1) / a.lse_chunk;
  const float2* p = a.partials + (int64_t)u * a.n_chunks * a.rows_max + row;
  float M = -INFINITY;
  for (int c = 0; c < n_chunks; ++c) M = fmaxf(M, p[(int64_t)c * a.rows_max].x);
  float S = 0.f;
  for (int c = 0; c < n_chunks; ++c) {
    float2 v = p[(int64_t)c * a.rows_max];
    if (v.x > -INFINITY) S += v.y * exp2f(v.x - M);
  }
  const float lse = (M + log2f(S)) * kLn2;
  const int w = row / G, g = row % G;
  const int64_t o = ((int64_t)slab * a.sum_win + w0 + w) * a.n_q_heads + h * G + g;
  lse_out[o] = lse;
}

}  // namespace actkv
