// actkv_budget: confidence monitor and budget update (Section 6.1, Algorithm 2).
//
// Token confidence T = logsumexp(z) - mean(top-k z) of every logits row, exact top-k whatever the distribution, no sort:
//   token_conf_cluster_kernel  few rows: a cluster of CTAs per row;
//   token_conf_sweep_kernel    many rows: one CTA per row, one sweep over HBM;
//   token_conf_exact           the rows these two give up on: one CTA, a 3-pass radix select (digits of 11, 11 and 10
//                              bits of the order-preserving integer image of the floats), one sweep from HBM, two from L2.
// trend_kernel — one CTA per request: append, window-min pooling, nearest-rank bottom-b%,
//   least-squares slope in float64, budget update with the optional integer clamp.
#include "common.cuh"

namespace actkv {

constexpr int TC_NT = 512;        // threads per CTA of the token-confidence kernels

__device__ __forceinline__ uint32_t okey(float x) {
  uint32_t b = __float_as_uint(x);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float okey_inv(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

__device__ __forceinline__ float block_reduce_max(float v, float* sm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if (lane == 0) sm[warp] = v;
  __syncthreads();
  float r = sm[0];
  for (int w = 1; w < (int)(blockDim.x >> 5); ++w) r = fmaxf(r, sm[w]);
  return r;
}

// Fixed-order tree: deterministic for a given block size.
__device__ __forceinline__ double block_reduce_sum(double v, double* sm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if (lane == 0) sm[warp] = v;
  __syncthreads();
  double r = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r += sm[w];
  return r;
}

// Finds the digit d with  #(digit > d) < remaining <= #(digit >= d)  in hist[0..nbins).
// All threads call it; results land in shared s_out[0] = d, s_out[1] = remaining - #(digit > d),
// s_out[2] = hist[d].
__device__ __forceinline__ void pick_digit(const uint32_t* hist, int nbins, uint32_t remaining,
                                           uint32_t* warp_tot, uint32_t* s_out) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // each thread owns `per` (at most 4) adjacent bins, descending from nbins - 1 - per * tid
  const int per = (nbins + (int)blockDim.x - 1) / (int)blockDim.x;
  const int b0 = nbins - 1 - per * tid;
  uint32_t v[4], mine = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int b = b0 - j;
    v[j] = (j < per && b >= 0) ? hist[b] : 0u;
    mine += v[j];
  }
  uint32_t incl = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    uint32_t t = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += t;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  uint32_t acc = incl - mine;                    // #(digit > b0)
  for (int w = 0; w < warp; ++w) acc += warp_tot[w];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int b = b0 - j;
    if (j < per && b >= 0 && acc < remaining && acc + v[j] >= remaining) {
      s_out[0] = (uint32_t)b; s_out[1] = remaining - acc; s_out[2] = v[j];
    }
    acc += v[j];
  }
  __syncthreads();
}

// Where a row's confidence goes.
struct ConfOut {
  const int32_t* tok_indptr;
  int32_t n_req;
  float* conf_hist;
  const int32_t* hist_len;
  int32_t hist_cap;
  int32_t* status;
};

// The place of row `row`: its request (the last r with tok_indptr[r] <= row) and the position in that request's history.
// One converged warp calls it early, so that its two round trips to memory run beside the row's own loads.
struct RowSlot {
  int r, pos;
};
__device__ __forceinline__ RowSlot find_slot(const ConfOut& out, int row) {
  const int lane = threadIdx.x & 31;
  int n = 0;                                     // requests 1 .. n_req - 1 that begin at or before the row
  for (int r = 1 + lane; r < out.n_req; r += 32) n += out.tok_indptr[r] <= row ? 1 : 0;
  n = (int)__reduce_add_sync(0xffffffffu, (uint32_t)n);
  return RowSlot{n, out.hist_len[n] + (row - out.tok_indptr[n])};
}
__device__ __forceinline__ void store_conf(const ConfOut& out, const RowSlot& at, float T) {
  if (at.pos < out.hist_cap) out.conf_hist[(int64_t)at.r * out.hist_cap + at.pos] = T;
  else report(out.status, ACTKV_E_INVALID, at.r, at.pos);
}

struct ExactSmem {
  uint32_t hist[2048];
  uint32_t warp_tot[TC_NT / 32];
  uint32_t s_pick[3];
  float red_f[TC_NT / 32];
  double red_d[TC_NT / 32];
};

// The three-sweep form, for the rows the other kernels give up on.  All TC_NT threads of the CTA call it; thread 0 has
// the result.
__device__ __noinline__ float token_conf_exact(const float* __restrict__ z, int vocab, int k, ExactSmem* sm) {
  uint32_t *hist = sm->hist, *warp_tot = sm->warp_tot, *s_pick = sm->s_pick;
  float* red_f = sm->red_f;
  double* red_d = sm->red_d;
  const int tid = threadIdx.x, lane = tid & 31;

  // ---- pass 1 (HBM): max, histogram of key bits 31..21 ------------------------------------
  for (int i = tid; i < 2048; i += TC_NT) hist[i] = 0;
  __syncthreads();
  float mx = -INFINITY;
  for (int i0 = 0; i0 < vocab; i0 += TC_NT) {
    const int i = i0 + tid;
    const bool in = i < vocab;
    const float x = in ? z[i] : 0.f;
    const uint32_t voters = __ballot_sync(0xffffffffu, in);
    if (in) {
      mx = fmaxf(mx, x);
      const uint32_t bin = okey(x) >> 21;
      const uint32_t peers = __match_any_sync(voters, bin);
      if (lane == (__ffs(peers) - 1)) atomicAdd(&hist[bin], (uint32_t)__popc(peers));
    }
  }
  mx = block_reduce_max(mx, red_f);             // includes the barrier that completes hist
  pick_digit(hist, 2048, (uint32_t)k, warp_tot, s_pick);
  const uint32_t d1 = s_pick[0];
  uint32_t remaining = s_pick[1];
  __syncthreads();

  // ---- pass 2 (L2): sum exp(z - max), histogram of bits 20..10 among keys with digit d1 -----
  for (int i = tid; i < 2048; i += TC_NT) hist[i] = 0;
  __syncthreads();
  double se = 0.0;
  {
    float se_f = 0.f;
    const float mx2 = mx * kLog2e;
    for (int i0 = 0; i0 < vocab; i0 += TC_NT) {
      const int i = i0 + tid;
      const bool in = i < vocab;
      const float x = in ? z[i] : 0.f;
      const uint32_t key = okey(x);
      const bool cand = in && (key >> 21) == d1;
      const uint32_t voters = __ballot_sync(0xffffffffu, cand);
      if (in) se_f += exp2f(fmaf(x, kLog2e, -mx2));
      if (cand) {
        const uint32_t bin = (key >> 10) & 2047u;
        const uint32_t peers = __match_any_sync(voters, bin);
        if (lane == (__ffs(peers) - 1)) atomicAdd(&hist[bin], (uint32_t)__popc(peers));
      }
    }
    se = (double)se_f;
  }
  se = block_reduce_sum(se, red_d);
  pick_digit(hist, 2048, remaining, warp_tot, s_pick);
  const uint32_t d2 = s_pick[0];
  remaining = s_pick[1];
  const uint32_t prefix22 = (d1 << 11) | d2;
  __syncthreads();

  // ---- pass 3 (L2): sum of logits above the 22-bit prefix, histogram of the last 10 bits ----
  for (int i = tid; i < 1024; i += TC_NT) hist[i] = 0;
  __syncthreads();
  double top = 0.0;
  for (int i0 = 0; i0 < vocab; i0 += TC_NT) {
    const int i = i0 + tid;
    const bool in = i < vocab;
    const float x = in ? z[i] : 0.f;
    const uint32_t key = okey(x);
    const uint32_t p22 = key >> 10;
    const bool cand = in && p22 == prefix22;
    const uint32_t voters = __ballot_sync(0xffffffffu, cand);
    if (in && p22 > prefix22) top += (double)x;
    if (cand) {
      const uint32_t bin = key & 1023u;
      const uint32_t peers = __match_any_sync(voters, bin);
      if (lane == (__ffs(peers) - 1)) atomicAdd(&hist[bin], (uint32_t)__popc(peers));
    }
  }
  top = block_reduce_sum(top, red_d);
  pick_digit(hist, 1024, remaining, warp_tot, s_pick);
  if (tid == 0) {
    const uint32_t d3 = s_pick[0];
    const uint32_t need = s_pick[1];
    // keys sharing the 22-bit prefix: value is fixed by the last digit, counts are in hist
    for (uint32_t b = 1023; b > d3; --b)
      if (hist[b]) top += (double)hist[b] * (double)okey_inv((prefix22 << 10) | b);
    top += (double)need * (double)okey_inv((prefix22 << 10) | d3);
    const float lse = mx + logf((float)se);
    return lse - (float)(top / (double)k);
  }
  return 0.f;
}

// -----------------------------------------------------------------------------------------------
// Single-sweep token confidence.  A lower bound tau of the row's k-th largest logit lets one sweep keep
// only the few logits >= tau while it sums the exponentials:
//  (A) the first SW_HEAD logits are split into 64 chunks; the k-th largest of the 64 chunk maxima is tau
//      (k of the row's logits are at least that large; k <= 64), the largest of them the reference M of
//      the exponentials;
//  (B) the row is streamed ONCE from HBM: sum of exp(x - M) per thread, logits >= tau appended to a shared
//      candidate list (about half a percent of the row);
//  (C) the top k of the list are the top k of the row: exact radix select in shared memory.
// Rows whose list overflows (adversarial order, e.g. ascending logits), whose sum overflows (M is not the
// row's maximum) or with k > 64 are redone by the same CTA in three sweeps.
// Two CTAs of 512 threads per SM: one streams while the other is in its serial phases.
constexpr int SW_HEAD = 4096;
constexpr int SW_CAP = 4096;
constexpr int SW_NT = TC_NT;
constexpr int SW_PER = SW_HEAD / SW_NT;     // head logits per thread (8: a chunk is 8 lanes x 8 = 64 logits)

struct SweepSmem {
  float cand[SW_CAP];
  float chunk_max[64];
  uint32_t n_cand;
  float tau, ref;
  ExactSmem ex;
};

// k-th largest (k >= 1) of vals[0..n) by three radix digits; all threads call it.  Returns the key of
// that element and the number of elements equal to it that belong to the top k.
__device__ __forceinline__ void smem_kth_largest(const float* vals, int n, uint32_t k, SweepSmem* sm,
                                                 uint32_t& key_out, uint32_t& need_out) {
  const int tid = threadIdx.x;
  uint32_t prefix = 0, remaining = k;
  for (int pass = 0; pass < 3; ++pass) {
    const int nb = pass == 2 ? 1024 : 2048;
    const int shift = pass == 0 ? 21 : (pass == 1 ? 10 : 0);
    for (int i = tid; i < nb; i += SW_NT) sm->ex.hist[i] = 0;
    __syncthreads();
    for (int i = tid; i < n; i += SW_NT) {
      const uint32_t key = okey(vals[i]);
      const bool in = pass == 0 || (pass == 1 ? (key >> 21) == prefix : (key >> 10) == prefix);
      if (in) atomicAdd(&sm->ex.hist[(key >> shift) & (uint32_t)(nb - 1)], 1u);
    }
    __syncthreads();
    pick_digit(sm->ex.hist, nb, remaining, sm->ex.warp_tot, sm->ex.s_pick);
    prefix = (pass == 0) ? sm->ex.s_pick[0] : ((prefix << (pass == 1 ? 11 : 10)) | sm->ex.s_pick[0]);
    remaining = sm->ex.s_pick[1];
    __syncthreads();
  }
  key_out = prefix;
  need_out = remaining;
}

__global__ void __launch_bounds__(SW_NT, 2) token_conf_sweep_kernel(
    const float* __restrict__ logits, int32_t vocab, int32_t k_top, const ConfOut out) {
  pdl_begin(logits);
  extern __shared__ __align__(16) uint8_t sweep_raw[];
  SweepSmem* sm = reinterpret_cast<SweepSmem*>(sweep_raw);
  const int row = blockIdx.x, tid = threadIdx.x;
  const float* z = logits + (int64_t)row * vocab;
  const int k = min(k_top, vocab);
  const int n_head = min(vocab, SW_HEAD);

  // ---- (A) threshold and reference from the chunk maxima of the head ----
  const bool vec = (vocab % 4 == 0) && ((reinterpret_cast<uintptr_t>(z) & 15) == 0);
  float hv[SW_PER];
  float hm = -INFINITY;
#pragma unroll
  for (int j = 0; j < SW_PER; ++j) {
    const int i = tid * SW_PER + j;
    hv[j] = (i < n_head) ? z[i] : -INFINITY;
  }
  RowSlot at{0, 0};
  if (tid < 32) at = find_slot(out, row);
#pragma unroll
  for (int j = 0; j < SW_PER; ++j) hm = fmaxf(hm, hv[j]);
#pragma unroll
  for (int o = 4; o >= 1; o >>= 1) hm = fmaxf(hm, __shfl_xor_sync(0xffffffffu, hm, o));     // over 8 lanes
  if ((tid & 7) == 0) sm->chunk_max[tid >> 3] = hm;
  if (tid == 0) sm->n_cand = 0;
  __syncthreads();
  if (tid < 64) {
    const float v = sm->chunk_max[tid];
    int rank = 0;                                            // chunk maxima that come before this one, descending
    float top = -INFINITY;
    for (int u = 0; u < 64; ++u) {
      const float w = sm->chunk_max[u];
      rank += (w > v || (w == v && u < tid)) ? 1 : 0;
      top = fmaxf(top, w);
    }
    if (rank == k - 1) sm->tau = v;
    if (tid == 0) sm->ref = top;
  }
  __syncthreads();
  const float tau = sm->tau, M = sm->ref;
  if (k > 64 || !(M > -INFINITY)) {                          // (uniform) no bound from 64 maxima: the fallback's row
    const float T = token_conf_exact(z, vocab, k, &sm->ex);
    if (tid == 0) store_conf(out, at, T);
    return;
  }

  // ---- (B) one sweep: sum of exp(x - M) per thread, candidates >= tau.  M is the maximum of the head, not
  //      of the row: later logits may exceed it (the sum may grow up to the float range; a row whose sum
  //      overflows is left to the fallback) ----
  const float nmc = -M * kLog2e;
  float s = 0.f;
  auto visit = [&](float x) {
    s += exp2f(fmaf(x, kLog2e, nmc));
    if (x >= tau) {
      const uint32_t pos = atomicAdd(&sm->n_cand, 1u);
      if (pos < SW_CAP) sm->cand[pos] = x;
    }
  };
#pragma unroll
  for (int j = 0; j < SW_PER; ++j)
    if (tid * SW_PER + j < n_head) visit(hv[j]);
  if (vec) {
    const float4* z4 = reinterpret_cast<const float4*>(z);
    const int n4 = vocab / 4;
    int i = SW_HEAD / 4 + tid;
    for (; i + 7 * SW_NT < n4; i += 8 * SW_NT) {               // eight 16-byte loads in flight per thread
      float4 v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = z4[i + j * SW_NT];
#pragma unroll
      for (int j = 0; j < 8; ++j) { visit(v[j].x); visit(v[j].y); visit(v[j].z); visit(v[j].w); }
    }
    for (; i < n4; i += SW_NT) {
      const float4 a = z4[i];
      visit(a.x); visit(a.y); visit(a.z); visit(a.w);
    }
  } else {
    for (int i = SW_HEAD + tid; i < vocab; i += SW_NT) visit(z[i]);
  }
  const double S = block_reduce_sum((double)s, sm->ex.red_d);   // fixed-order tree
  __syncthreads();
  const uint32_t n_cand = sm->n_cand;
  if (n_cand > SW_CAP || !(S < 3.0e38)) {                    // adversarial order or overflow: the fallback's row
    const float T = token_conf_exact(z, vocab, k, &sm->ex);
    if (tid == 0) store_conf(out, at, T);
    return;
  }
  // ---- (C) the top k of the candidates are the top k of the row ----
  const uint32_t n_all = n_cand;
  uint32_t kth_key, need_k;
  smem_kth_largest(sm->cand, (int)n_all, (uint32_t)k, sm, kth_key, need_k);
  const float kth = okey_inv(kth_key);
  double top = 0.0;
  for (int i = tid; i < (int)n_all; i += SW_NT) {
    const float x = sm->cand[i];
    if (okey(x) > kth_key) top += (double)x;
  }
  top = block_reduce_sum(top, sm->ex.red_d);
  if (tid == 0) {
    top += (double)need_k * (double)kth;
    const float lse = M + logf((float)S);
    store_conf(out, at, lse - (float)(top / (double)k));
  }
}

// -----------------------------------------------------------------------------------------------
// A row over a cluster of CTAs, for calls of few rows (one decode step adds one row per request): every CTA takes its
// share of the row into registers with all its loads in flight at once, so that a row costs about one memory round trip
// and a few dozen rows keep the chip busy.
// It is bound by latency: 12 us for 16 rows of 151936 (9.7 MB), where one CTA per row took 23.
// Each CTA: its maximum M_c, sum of exp(x - M_c), and a bound tau on its own k-th largest logit (the k-th largest of 64
// chunk maxima), logits >= tau into a shared list (some 25 of them).  The first CTA of the cluster gathers the lists
// through distributed shared memory, ranks them (larger first, equal values being interchangeable) and adds the top k in
// rank order.  Rows it cannot take (k > 64, a list that overflows, fewer than k finite logits) are redone by that CTA in
// three sweeps.
constexpr int CL_CAP = 512;                 // candidates of one CTA
constexpr int CL_MAX = 8;                   // CTAs of a cluster
constexpr int CL_CTAS = 4 * 148;            // CTAs of a launch
struct ClusterSmem {
  float cand[CL_CAP];
  float all[CL_MAX * CL_CAP];
  float top[64];
  float chunk_max[64];
  float warp_sum[TC_NT / 32];
  float m, tau;
  double s;
  uint32_t n;
  int give_up;
  ExactSmem ex;
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// p: an address in this CTA's shared memory; the same place in CTA `rank` of the cluster
template <class T>
__device__ __forceinline__ uint32_t remote_addr(const T* p, uint32_t rank) {
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return ra;
}
__device__ __forceinline__ uint32_t remote(const uint32_t* p, uint32_t rank) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(remote_addr(p, rank)) : "memory");
  return v;
}
__device__ __forceinline__ float remote(const float* p, uint32_t rank) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(remote_addr(p, rank)) : "memory");
  return v;
}
__device__ __forceinline__ double remote(const double* p, uint32_t rank) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(remote_addr(p, rank)) : "memory");
  return v;
}

// NV: 16-byte vectors per thread.  Vectors are aligned whatever the row's alignment; the elements of the first and last
// one that belong to the neighbouring rows are not read.
template <int NV>
__global__ void __launch_bounds__(TC_NT) token_conf_cluster_kernel(const float* __restrict__ logits, int32_t vocab,
                                                                   int32_t k_top, int32_t n_parts, int32_t vecs_per_part,
                                                                   const ConfOut out) {
  pdl_begin(logits);
  __shared__ ClusterSmem sm;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int row = blockIdx.x / n_parts;
  const uint32_t part = cluster_rank();
  const float* z = logits + (int64_t)row * vocab;
  const int k = min(k_top, vocab);
  const int mis = (int)((reinterpret_cast<uintptr_t>(z) >> 2) & 3u);     // elements between the vector boundary and the row
  const float* zb = z - mis;
  const int v_end = min((int)(part + 1) * vecs_per_part, (mis + vocab + 3) / 4);
  float x[4 * NV];
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    const int v = (int)part * vecs_per_part + tid + j * TC_NT;
    float4 q = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    if (v < v_end) {
      if (4 * v >= mis && 4 * v + 4 <= mis + vocab) {
        q = __ldg(reinterpret_cast<const float4*>(zb) + v);
      } else {
        if (4 * v >= mis && 4 * v < mis + vocab) q.x = __ldg(zb + 4 * v);
        if (4 * v + 1 >= mis && 4 * v + 1 < mis + vocab) q.y = __ldg(zb + 4 * v + 1);
        if (4 * v + 2 >= mis && 4 * v + 2 < mis + vocab) q.z = __ldg(zb + 4 * v + 2);
        if (4 * v + 3 >= mis && 4 * v + 3 < mis + vocab) q.w = __ldg(zb + 4 * v + 3);
      }
    }
    x[4 * j] = q.x; x[4 * j + 1] = q.y; x[4 * j + 2] = q.z; x[4 * j + 3] = q.w;
  }
  RowSlot at{0, 0};
  if (part == 0 && warp == 0) at = find_slot(out, row);
  if (tid == 0) { sm.n = 0u; sm.tau = -INFINITY; }
  float hm = -INFINITY;
#pragma unroll
  for (int i = 0; i < 4 * NV; ++i) hm = fmaxf(hm, x[i]);
#pragma unroll
  for (int o = 4; o >= 1; o >>= 1) hm = fmaxf(hm, __shfl_xor_sync(0xffffffffu, hm, o));
  if ((tid & 7) == 0) sm.chunk_max[tid >> 3] = hm;
  __syncthreads();
  if (tid < 64) {
    const float v = sm.chunk_max[tid];
    int rank = 0;
    float top = -INFINITY;
#pragma unroll 16
    for (int u = 0; u < 64; ++u) {
      const float w = sm.chunk_max[u];
      rank += (w > v || (w == v && u < tid)) ? 1 : 0;
      top = fmaxf(top, w);
    }
    if (rank == k - 1) sm.tau = v;
    if (tid == 0) sm.m = top;
  }
  __syncthreads();
  const float tau = sm.tau, M = sm.m;
  const float nmc = M > -INFINITY ? -M * kLog2e : 0.f;
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < 4 * NV; ++i) {
    s += exp2f(fmaf(x[i], kLog2e, nmc));
    if (x[i] >= tau && x[i] > -INFINITY) {
      const uint32_t pos = atomicAdd(&sm.n, 1u);
      if (pos < CL_CAP) sm.cand[pos] = x[i];
    }
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) sm.warp_sum[warp] = s;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < TC_NT / 32; ++w) t += (double)sm.warp_sum[w];
    sm.s = t;
  }
  cluster_sync();
  if (part == 0) {
    // lane c of every warp has what CTA c of the cluster found
    const bool mine = lane < n_parts;
    const uint32_t n_c = mine ? remote(&sm.n, lane) : 0u;
    const float m_c = mine ? remote(&sm.m, lane) : -INFINITY;
    const double s_c = mine && warp == 0 ? remote(&sm.s, lane) : 0.0;
    const bool bad = k > 64 || __any_sync(0xffffffffu, n_c > (uint32_t)CL_CAP);
    const uint32_t total = __reduce_add_sync(0xffffffffu, n_c);
    const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? n_c : 0u);
    float Mr = m_c;
#pragma unroll
    for (int o = CL_MAX / 2; o >= 1; o >>= 1) Mr = fmaxf(Mr, __shfl_xor_sync(0xffffffffu, Mr, o));
    Mr = __shfl_sync(0xffffffffu, Mr, 0);
    float T;
    if (!bad && Mr > -INFINITY && (int)total >= k) {   // (the same for every thread)
      if (warp < n_parts) {                            // a warp per list
        const uint32_t n = __shfl_sync(0xffffffffu, n_c, warp);
        for (uint32_t i = lane; i < n; i += 32) sm.all[before + i] = remote(&sm.cand[i], warp);
      }
      if (tid < 64) sm.top[tid] = 0.f;
      __syncthreads();
      for (uint32_t i = tid; i < total; i += TC_NT) {
        const float v = sm.all[i];
        int rank = 0;
#pragma unroll 8
        for (uint32_t j = 0; j < total; ++j) {
          const float w = sm.all[j];
          rank += (w > v || (w == v && j < i)) ? 1 : 0;
        }
        if (rank < k) sm.top[rank] = v;
      }
      __syncthreads();
      if (warp == 0) {
        double S = m_c > -INFINITY ? s_c * (double)exp2f((m_c - Mr) * kLog2e) : 0.0;
        double top = (double)sm.top[lane] + (double)sm.top[lane + 32];
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) {
          S += __shfl_xor_sync(0xffffffffu, S, o);
          top += __shfl_xor_sync(0xffffffffu, top, o);
        }
        T = Mr + logf((float)S) - (float)(top / (double)k);
      }
    } else {
      T = token_conf_exact(z, vocab, k, &sm.ex);
    }
    if (tid == 0) store_conf(out, at, T);
  }
  cluster_sync();                                      // the lists stay until the first CTA has read them
}

struct BudgetParamsDev {
  int32_t w, s;
  double b_percent, scale_up;
  int32_t B_upper, clamp_lo_ppm, clamp_hi_ppm;
};

constexpr int TR_NT = 256;
constexpr int TR_CAP = 4096;                // pooled values kept in shared memory (longer sequences: the workspace)

// One CTA per request, every phase over the whole CTA.
// It is bound by the chain of its phases: 6.5 us at a history of 512 tokens (26 us when one thread walked the windows
// and the bins of every digit; 74 -> 35 us for a whole call at 2900 tokens).
__global__ void __launch_bounds__(TR_NT) trend_kernel(
    const int32_t* __restrict__ tok_indptr, const float* __restrict__ conf_hist, int32_t* hist_len,
    int32_t hist_cap, BudgetParamsDev p, const int32_t* __restrict__ seq_len,
    const int32_t* __restrict__ budget_in, int32_t* __restrict__ budget_out, double* slope_out,
    float* pooled_ws, int32_t max_m) {
  pdl_begin(tok_indptr, conf_hist, seq_len, budget_in);
  static_assert(TR_NT == 256, "one thread per bin of a digit");
  __shared__ float s_pool[TR_CAP], s_block[TR_CAP];
  __shared__ uint32_t s_hist[256];
  __shared__ uint32_t s_prefix, s_remaining;
  __shared__ uint32_t s_warp[TR_NT / 32];
  __shared__ double s_red[TR_NT / 32];
  const int r = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n_new = tok_indptr ? tok_indptr[r + 1] - tok_indptr[r] : 0;
  const int Lh = min(hist_cap, hist_len[r] + n_new);
  const float* TL = conf_hist + (int64_t)r * hist_cap;
  const int M = (Lh >= p.w) ? (Lh - p.w) / p.s + 1 : 0;
  float* Rp = M <= TR_CAP ? s_pool : pooled_ws + (int64_t)r * max_m;
  const int bpw = p.w / p.s;                            // blocks of s values per window when s divides w
  if (p.w % p.s == 0 && M + bpw - 1 <= TR_CAP) {
    // minima of the blocks of s values that the windows share, then of the bpw blocks of a window
    for (int j = tid; M > 0 && j < M + bpw - 1; j += TR_NT) {
      float v = TL[j * p.s];
#pragma unroll 8
      for (int i = 1; i < p.s; ++i) v = fminf(v, TL[j * p.s + i]);
      s_block[j] = v;
    }
    __syncthreads();
    for (int m = tid; m < M; m += TR_NT) {
      float v = s_block[m];
      for (int i = 1; i < bpw; ++i) v = fminf(v, s_block[m + i]);
      Rp[m] = v;
    }
  } else {
    for (int m = tid; m < M; m += TR_NT) {
      float v = TL[m * p.s];
      for (int i = 1; i < p.w; ++i) v = fminf(v, TL[m * p.s + i]);
      Rp[m] = v;
    }
  }
  __syncthreads();
  double alpha = 0.0;
  if (M > 0) {
    int rank = (int)ceil(p.b_percent * (double)M / 100.0);
    if (rank < 1) rank = 1;
    if (rank > M) rank = M;
    // nearest-rank percentile: the rank-th smallest value, i.e. the v with #(< v) < rank <= #(<= v), by a radix
    // select over the order-preserving integer image of the values (four 8-bit digits, most significant first):
    // 4 M steps for any history length (counting the values below each candidate would take M^2)
    if (tid == 0) { s_prefix = 0u; s_remaining = (uint32_t)rank; }
    for (int pass = 0; pass < 4; ++pass) {
      const int shift = 24 - 8 * pass;
      const uint32_t himask = pass == 0 ? 0u : (0xffffffffu << (shift + 8));
      s_hist[tid] = 0u;
      __syncthreads();
      const uint32_t prefix = s_prefix, rem = s_remaining;
      for (int m = tid; m < M; m += TR_NT) {
        const uint32_t k = okey(Rp[m]);
        if ((k & himask) == prefix) atomicAdd(&s_hist[(k >> shift) & 255u], 1u);
      }
      __syncthreads();
      const uint32_t mine = s_hist[tid];
      uint32_t incl = mine;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
      }
      if (lane == 31) s_warp[warp] = incl;
      __syncthreads();
      for (int w = 0; w < warp; ++w) incl += s_warp[w];
      // ascending: the digit that holds the rem-th smallest
      if (incl - mine < rem && incl >= rem) { s_prefix = prefix | ((uint32_t)tid << shift); s_remaining = rem - (incl - mine); }
      __syncthreads();
    }
    const float qv = okey_inv(s_prefix);
    // R = values <= q in time order; least-squares slope in float64 against their positions 0 .. n - 1, whose mean (n - 1) / 2 and
    // sum of squared deviations n (n^2 - 1) / 12 are known.  The deviations of the positions add up to nothing, so the values
    // themselves are summed: a product of a half-integer and a float is exact, and so are the sums of some ten thousand of them.
    // A slope that is zero comes out as zero, whatever the order (the budget follows its sign; with the values' deviations from their
    // rounded mean it was noise of either sign).
    int n = 0;
    for (int m = tid; m < M; m += TR_NT) n += Rp[m] <= qv ? 1 : 0;
    n = (int)block_reduce_sum((double)n, s_red);
    if (n >= 2) {
      const double xm = (double)(n - 1) * 0.5;
      double sxy = 0.0;
      int before = 0;                                   // values of R in earlier rounds of TR_NT
      for (int m0 = 0; m0 < M; m0 += TR_NT) {
        const int m = m0 + tid;
        const bool in = m < M && Rp[m] <= qv;
        const uint32_t bal = __ballot_sync(0xffffffffu, in);
        __syncthreads();
        if (lane == 0) s_warp[warp] = (uint32_t)__popc(bal);
        __syncthreads();
        int i = before + __popc(bal & ((1u << lane) - 1u));
        for (int w = 0; w < TR_NT / 32; ++w) {
          if (w < warp) i += (int)s_warp[w];
          before += (int)s_warp[w];
        }
        if (in) sxy += ((double)i - xm) * (double)Rp[m];
      }
      sxy = block_reduce_sum(sxy, s_red);
      // (infinite values have no slope)
      alpha = fabs(sxy) < (double)INFINITY ? sxy / ((double)n * ((double)n * (double)n - 1.0) / 12.0) : (double)NAN;
    }
  }
  if (tid == 0) {
    long long B = budget_in[r];
    if (alpha < 0.0) {
      double scaled = floor((double)B * p.scale_up);
      long long Bs = (long long)scaled;
      B = Bs < (long long)p.B_upper ? Bs : (long long)p.B_upper;
    }
    if (p.clamp_hi_ppm > 0 && seq_len != nullptr) {
      const long long L = seq_len[r];
      const long long lo = (L * p.clamp_lo_ppm + 999999LL) / 1000000LL;
      const long long hi = (L * p.clamp_hi_ppm) / 1000000LL;
      if (B < lo) B = lo;
      if (B > hi) B = hi;
    }
    budget_out[r] = (int32_t)B;
    if (slope_out) slope_out[r] = alpha;
    hist_len[r] = Lh;
  }
}

template <int NV>
static int launch_cluster(const float* logits, int32_t vocab, int32_t n_rows, int32_t k, int parts, int vecs, const ConfOut& out,
                          cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n_rows * parts));
  cfg.blockDim = dim3(TC_NT);
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)parts;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  if (cudaLaunchKernelEx(&cfg, token_conf_cluster_kernel<NV>, logits, vocab, k, (int32_t)parts, (int32_t)vecs, out) != cudaSuccess) {
    (void)cudaGetLastError();
    return ACTKV_E_CUDA;
  }
  return ACTKV_OK;
}

static int launch_token_conf(const float* logits, int32_t vocab, int32_t n_rows, int32_t k, const ConfOut& out, cudaStream_t s) {
  // A cluster per row up to four CTAs per SM, i.e. one or two rounds of clusters; beyond that the work that every CTA
  // adds (its own chunk maxima, list and barriers) costs more than the shorter rows save.  Whole call, 151936 logits per
  // row, clusters against one CTA per row: 1 row 20 / 33 us, 16 rows 24 / 34, 48 rows 35 / 39, 64 rows 38 / 40,
  // 128 rows 66 / 42.
  const int vecs_all = vocab / 4 + 2;                  // vectors a row of any alignment touches
  int parts = 1;
  while (parts < CL_MAX && vecs_all / parts > 4 * TC_NT) parts <<= 1;
  const int vecs = (vecs_all + parts - 1) / parts, per_thread = (vecs + TC_NT - 1) / TC_NT;
  if ((int64_t)n_rows * parts <= CL_CTAS && per_thread <= 16) {
    if (per_thread <= 4) return launch_cluster<4>(logits, vocab, n_rows, k, parts, vecs, out, s);
    if (per_thread <= 10) return launch_cluster<10>(logits, vocab, n_rows, k, parts, vecs, out, s);
    return launch_cluster<16>(logits, vocab, n_rows, k, parts, vecs, out, s);
  }
  const size_t sm = sizeof(SweepSmem);
  if (ensure_dyn_smem(token_conf_sweep_kernel, sm) != cudaSuccess) return ACTKV_E_CUDA;
  launch_pdl(token_conf_sweep_kernel, (unsigned)n_rows, SW_NT, sm, s, logits, vocab, k, out);
  ACTKV_CHECK_LAUNCH();
  return ACTKV_OK;
}

}  // namespace actkv

extern "C" {

size_t actkv_budget_workspace_bytes(int32_t n_rows, int32_t n_req, int32_t hist_cap) {
  if (n_rows < 0 || n_req < 0 || hist_cap < 0) return 0;
  // one pooled sequence of at most hist_cap values per request, behind 4 bytes per row that no kernel uses (the confidences go
  // straight into the history; callers have sized their workspaces by this figure)
  return actkv::align_up((size_t)n_rows * 4, 256) + actkv::align_up((size_t)n_req * hist_cap * 4, 256);
}

int actkv_budget(const float* logits, const int32_t* tok_indptr, int32_t n_rows, int32_t vocab,
                 float* conf_hist, int32_t* hist_len, int32_t hist_cap,
                 const actkv_budget_params_t* params, const int32_t* seq_len,
                 const int32_t* budget_in, int32_t* budget_out, double* slope_out, int32_t n_req,
                 void* ws, size_t ws_bytes, int32_t* status, actkv_stream_t stream) {
  if (!params || n_req < 0 || n_rows < 0 || hist_cap <= 0 || hist_cap > 65536) return ACTKV_E_INVALID;
  if (params->k <= 0 || params->w <= 0 || params->s <= 0 || !(params->b_percent >= 0.0)) return ACTKV_E_INVALID;
  if (n_req == 0) return ACTKV_OK;
  if (!conf_hist || !hist_len || !budget_in || !budget_out || !ws) return ACTKV_E_INVALID;
  if (n_rows > 0 && (!logits || !tok_indptr || vocab <= 0)) return ACTKV_E_INVALID;
  if (params->clamp_hi_ppm > 0 && !seq_len) return ACTKV_E_INVALID;
  if (ws_bytes < actkv_budget_workspace_bytes(n_rows, n_req, hist_cap)) return ACTKV_E_WORKSPACE;
  cudaStream_t s = (cudaStream_t)stream;
  float* pooled = (float*)((char*)ws + actkv::align_up((size_t)n_rows * 4, 256));
  if (n_rows > 0) {
    const int rc = actkv::launch_token_conf(logits, vocab, n_rows, params->k,
                                            actkv::ConfOut{tok_indptr, n_req, conf_hist, hist_len, hist_cap, status}, s);
    if (rc != ACTKV_OK) return rc;
  }
  actkv::BudgetParamsDev p{params->w, params->s, params->b_percent, params->scale_up,
                           params->B_upper, params->clamp_lo_ppm, params->clamp_hi_ppm};
  const int32_t max_m = hist_cap;
  actkv::launch_pdl(actkv::trend_kernel, (unsigned)n_req, actkv::TR_NT, 0, s,
                    n_rows > 0 ? tok_indptr : nullptr, conf_hist, hist_len, hist_cap, p, seq_len, budget_in, budget_out, slope_out, pooled, max_m);
  ACTKV_CHECK_LAUNCH();
  return ACTKV_OK;
}

}  // extern "C"
