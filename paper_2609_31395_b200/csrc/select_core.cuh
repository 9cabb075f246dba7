// TopK(score, k = B) for one unit held by one CTA (Algorithm 1 step 5), on order-preserving 32-bit keys.  Shared by
// actkv_select and the fused keep-score + select kernel.
//
// The n-th largest key is found by histograms whose bins divide the range that is still in question evenly:
// [smallest, largest key] first, then the bin that holds the n-th largest key.  Keys being float bits, the first bins
// are a fixed fraction of the scores' own octaves, so a warp's 32 increments fall into as many bins (fixed digits of
// the key put a unit's scores into a few dozen bins, and the increments of a warp onto one another).  One level leaves
// a few dozen keys, which are ranked against one another; degenerate score sets (ties, outliers) take more levels.
// The kept token indices then go out in ascending order, a contiguous segment of the unit per warp: count, one scan
// over the warps, emit.  Entries equal to the threshold are kept lowest index first.
#pragma once

#include "common.cuh"

namespace actkv {

constexpr int SEL_LIST = 160;           // keys that are ranked against one another (more: another histogram)

__device__ __forceinline__ uint32_t order_key(float x) {
  uint32_t b = __float_as_uint(x);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);     // larger float -> larger key
}
__device__ __forceinline__ float key_to_float(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

template <int NT>
struct SelectShared {
  uint32_t lo[NT / 32], hi[NT / 32];
  uint32_t warp_tot[NT / 32], warp_eq[NT / 32];
  uint32_t list[SEL_LIST];
  uint32_t n_list, bin, remaining, count, thr, need_eq, eq_total;
};

// [smallest, largest] over the CTA of per-thread ranges; contains a barrier.
template <int NT>
__device__ __forceinline__ void block_range(SelectShared<NT>& sh, uint32_t& lo, uint32_t& hi) {
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if ((threadIdx.x & 31) == 0) { sh.lo[threadIdx.x >> 5] = lo; sh.hi[threadIdx.x >> 5] = hi; }
  __syncthreads();
  const int w = threadIdx.x & (NT / 32 - 1);
  lo = __reduce_min_sync(0xffffffffu, sh.lo[w]);
  hi = __reduce_max_sync(0xffffffffu, sh.hi[w]);
}

// shift that maps [0, span] into fewer than `bins` (a power of two) values
__device__ __forceinline__ int bin_shift(uint32_t span, int bins) { return max(0, (32 - __clz((int)span)) - (31 - __clz(bins))); }

// Exclusive sum over the threads before this one in the CTA (thread 0 first); contains a barrier.
template <int NT, class T>
__device__ __forceinline__ T block_exclusive(T mine, T* warp_tot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T incl = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const T t = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += t;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  T before = lane < warp && lane < NT / 32 ? warp_tot[lane] : (T)0;
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) before += __shfl_xor_sync(0xffffffffu, before, d);
  return before + incl - mine;
}

// key_at(i), i < L: the unit's keys, n_above of them above hi, the others within [lo, hi]; hist: shared, BINS entries;
// n_above < n <= L.
// All NT threads call it; shared memory that key_at reads must be visible to them.
template <int NT, int BINS, class KeyAt>
__device__ __forceinline__ void select_and_emit(KeyAt key_at, uint32_t* hist, SelectShared<NT>& sh, uint32_t lo, uint32_t hi,
                                                int L, int n, int32_t* out, uint32_t* mask_row, int base, actkv_tie_t* tie,
                                                int u, int n_above = 0) {
  constexpr int WARPS = NT / 32, PER = BINS / NT;
  static_assert(BINS % NT == 0 && PER >= 1, "bins per thread");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t span = hi - lo, remaining = (uint32_t)(n - n_above);
  for (;;) {
    const int shift = bin_shift(span, BINS);
    for (int i = tid; i < BINS; i += NT) hist[i] = 0u;
    if (tid == 0) sh.n_list = 0u;
    __syncthreads();
    for (int i = tid; i < L; i += NT) {
      const uint32_t d = key_at(i) - lo;
      if (d <= span) atomicAdd(&hist[d >> shift], 1u);
    }
    __syncthreads();
    // sums over the bins, descending: thread t owns bins BINS - 1 - PER t .. BINS - PER - PER t
    const int b0 = BINS - PER * (tid + 1);
    uint32_t h[PER], mine = 0u;
#pragma unroll
    for (int j = 0; j < PER; ++j) { h[j] = hist[b0 + j]; mine += h[j]; }
    uint32_t acc = block_exclusive<NT, uint32_t>(mine, sh.warp_tot);
    if (acc < remaining && acc + mine >= remaining) {     // exactly one thread
#pragma unroll
      for (int j = PER - 1; j >= 0; --j) {
        if (acc < remaining && acc + h[j] >= remaining) {
          sh.bin = (uint32_t)(b0 + j);
          sh.remaining = remaining - acc;
          sh.count = h[j];
        }
        acc += h[j];
      }
    }
    __syncthreads();
    remaining = sh.remaining;
    lo += sh.bin << shift;
    span = min((1u << shift) - 1u, hi - lo);              // (the last bin may reach past hi, where the n_above keys lie)
    const uint32_t count = sh.count;
    if (shift == 0) {                                     // a bin is one key
      if (tid == 0) { sh.thr = lo; sh.need_eq = remaining; sh.eq_total = count; }
      break;
    }
    if (count <= (uint32_t)SEL_LIST) {
      for (int i = tid; i < L; i += NT) {
        const uint32_t k = key_at(i);
        if (k - lo <= span) sh.list[atomicAdd(&sh.n_list, 1u)] = k;
      }
      __syncthreads();
      for (uint32_t i = tid; i < count; i += NT) {
        const uint32_t v = sh.list[i];
        uint32_t above = 0u, equal = 0u;
#pragma unroll 4
        for (uint32_t j = 0; j < count; ++j) {
          const uint32_t w = sh.list[j];
          above += w > v;
          equal += w == v;
        }
        if (above < remaining && above + equal >= remaining) {   // (every entry of that value: the same words)
          sh.thr = v;
          sh.need_eq = remaining - above;
          sh.eq_total = equal;
        }
      }
      break;
    }
    __syncthreads();
  }
  __syncthreads();
  const uint32_t thr = sh.thr, need_eq = sh.need_eq;

  // ---- emit: warp w owns the indices [w seg, (w + 1) seg) ----
  const int seg = ((L + WARPS - 1) / WARPS + 31) & ~31;
  const int i_begin = warp * seg, i_end = min(L, i_begin + seg);
  uint32_t n_gt = 0u, n_eq = 0u;
#pragma unroll 4
  for (int i = i_begin + lane; i < i_end; i += 32) {
    const uint32_t k = key_at(i);
    n_gt += k > thr;
    n_eq += k == thr;
  }
  n_gt = __reduce_add_sync(0xffffffffu, n_gt);
  n_eq = __reduce_add_sync(0xffffffffu, n_eq);
  if (lane == 0) { sh.warp_tot[warp] = n_gt; sh.warp_eq[warp] = n_eq; }
  __syncthreads();
  uint32_t gt_before = __reduce_add_sync(0xffffffffu, lane < warp && lane < WARPS ? sh.warp_tot[lane] : 0u);
  uint32_t eq_before = __reduce_add_sync(0xffffffffu, lane < warp && lane < WARPS ? sh.warp_eq[lane] : 0u);
  const uint32_t below = (1u << lane) - 1u;
#pragma unroll 2
  for (int i0 = i_begin; i0 < i_end; i0 += 32) {
    const int i = i0 + lane;
    const uint32_t k = i < i_end ? key_at(i) : 0u;
    const bool gt = i < i_end && k > thr, eq = i < i_end && k == thr;
    const uint32_t m_gt = __ballot_sync(0xffffffffu, gt), m_eq = __ballot_sync(0xffffffffu, eq);
    const uint32_t e = eq_before + __popc(m_eq & below);  // entries equal to the threshold before this one
    if (gt || (eq && e < need_eq)) {
      out[gt_before + __popc(m_gt & below) + min(e, need_eq)] = i;
      if (mask_row) atomicOr(&mask_row[(base + i) >> 5], 1u << ((base + i) & 31));
    }
    gt_before += __popc(m_gt);
    eq_before += __popc(m_eq);
  }
  if (tie != nullptr && tid == 0) tie[u] = actkv_tie_t{key_to_float(thr), (int32_t)need_eq, (int32_t)sh.eq_total, n};
}

// Dynamic shared memory of a CTA that keeps a unit of max_tok keys beside `fixed` bytes, or as many keys as fit.
constexpr size_t SEL_SMEM_MAX = 232448 - 5120;           // (the rest: the static shared memory of the two kernels)
inline size_t resident_smem(size_t fixed, int64_t max_tok) {
  const size_t want = fixed + (size_t)(max_tok < 0 ? 0 : max_tok) * 4;
  return want < SEL_SMEM_MAX ? want : SEL_SMEM_MAX;
}

// Threads per unit for units of up to max_tok keys: 1024 where the sweeps are the latency, that is for long units and for few
// of them; 256 and 512 where several such CTAs fill an SM; 256 for units too short to occupy more, however few.  Keep-score update + TopK, against 1024 threads
// throughout: 2048 units of 1500 keys 48 / 119 us, 1024 of 3000 40 / 75, 1024 of 6000 68 / 107, 1024 of 16000 154 / 183,
// 200 of 20000 57 / 66; 64 units of 3000 keys 17 us with 256 threads, 13 with 1024.
inline int select_threads(int64_t units, int64_t max_tok) {
  if (max_tok <= (units > 148 ? 8192 : 1500)) return 256;
  if (units > 148 && max_tok <= 24000) return 512;
  return 1024;
}

// actkv_select with a bound on the unit lengths: checks the arguments and launches the kernel (select.cu).
int select_launch(const float* score, const int32_t* tok_indptr, int32_t sum_tok, int32_t max_tok, const int32_t* budget,
                  int32_t n_outer, int32_t n_req, const int32_t* keep_indptr, int32_t* sel_idx, int64_t sel_stride,
                  uint32_t* keep_mask, actkv_tie_t* tie_report, int32_t* status, cudaStream_t stream);

}  // namespace actkv
