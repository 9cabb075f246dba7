// actkv_keepscore: attention-aware LRFU keep-score (Section 5.1 equation; Algorithm 1 steps 2-4) and
// actkv_gather_f32 (the keep-scores of the survivors move with them, Algorithm 1 step 5 returns KS').
//
// Per (layer x KV head, request) unit, one CTA:
//   1. mass m_i = floor(clip(score_i, 0, 256) * 2^32) as 64-bit integers; total = sum m_i (exact);
//   2. mark = ceil(p_q * total / 10000); histograms of the integer mass over ever smaller key ranges (even bins, as
//      in select_core.cuh) and a ranking of the last few entries find the threshold score T with
//      mass(score > T) < mark <= mass(score >= T) — exact, independent of summation order;
//   3. entries above T are hits; of the entries equal to T the first ceil((mark - mass_above)/m_T)
//      by index are hits (the index of the last one is looked up only when not all of them are);
//   4. KS = lambda*KS + score*[hit], one float32 rounding per operation; the score buffer is
//      overwritten with the ranking key: KS, or +inf for the protected prefix.
#include "select_core.cuh"

namespace actkv {

constexpr int KS_BINS = 2048;
constexpr int KS_LIST = 256;             // entries that are ranked against one another

__device__ __forceinline__ unsigned long long ks_mass(float x) {
  const float c = fminf(fmaxf(x, 0.f), 256.f);
  return __float2ull_rz(c * 4294967296.f);               // exact: a power-of-two scaling, then truncation
}

// IEEE single-precision product and sum, one rounding each, subnormals kept whatever the build's
// flush-to-zero setting is (the recurrence decays towards them).
__device__ __forceinline__ float mul_ieee(float a, float b) {
  float d;
  asm("mul.rn.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ float add_ieee(float a, float b) {
  float d;
  asm("add.rn.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}

// (chunk sums stay below 2^32 for units of up to 2^17 entries; the total mass needs 2^16 or fewer, see below)
// What the fused form needs of actkv_select's arguments.
struct FusedSelectArgs {
  const int32_t* budget;
  const int32_t* keep_indptr;
  int32_t* sel_idx;
  int64_t sel_stride;
  uint32_t* keep_mask;
  actkv_tie_t* tie;
  int32_t* status;
};

template <int NT>
struct KeepShared {
  SelectShared<NT> sel;
  unsigned long long warp_tot[NT / 32];
  unsigned long long mass[KS_LIST];      // of the entries in `list`
  uint32_t list[KS_LIST];                // (sel.list, of SEL_LIST entries, is too short)
  unsigned long long above;
  uint32_t bin, thr, eq_total;
  int32_t last_tie;
};

// FUSED: the ranking keys go straight into TopK (select_core.cuh, on the keys in shared memory) instead of back to the
// score array: one read of the scores, one launch.  A unit longer than the host's bound does not fit in shared memory: its scores
// and keep-scores are read again for every sweep.
// What bounds it: latency, as in select.cu.  64 units x 16 requests of 8K-24K tokens 318 -> 146 us, 512 units of 35000
// 328 -> 202 us (fixed digits of 12, 12 and 8 bits and two ordered sweeps with block scans before).
template <bool FUSED, int NT>
__global__ void __launch_bounds__(NT) keepscore_kernel(
    float* __restrict__ score, const int32_t* __restrict__ tok_indptr, int32_t sum_tok, int32_t n_req,
    int32_t p_q, float lambda, const int32_t* __restrict__ n_protect, float* __restrict__ keep_score,
    uint32_t* __restrict__ hit_mask, int32_t cap, FusedSelectArgs fs) {
  pdl_begin(tok_indptr, n_protect);
  constexpr int WARPS = NT / 32, PER = KS_BINS / NT;
  // A mass is below 2^41; its three 14-bit chunks are summed in three 32-bit histograms (native shared
  // atomics; a 64-bit shared atomic is a compare-and-swap loop) and put together when the bins are scanned.  A chunk
  // of zeros, as most masses have, is not added.
  extern __shared__ __align__(16) uint32_t ks_smem[];
  __shared__ KeepShared<NT> sh;
  uint32_t* hist = ks_smem;                                            // [3][KS_BINS] mass chunks per bin
  uint32_t* skeys = ks_smem + 3 * KS_BINS;                             // [cap] order keys of the unit
  auto hist_add = [&](uint32_t bin, unsigned long long m) {
    const uint32_t c0 = (uint32_t)m & 0x3fffu, c1 = (uint32_t)(m >> 14) & 0x3fffu, c2 = (uint32_t)(m >> 28);
    if (c0) atomicAdd(&hist[bin], c0);
    if (c1) atomicAdd(&hist[KS_BINS + bin], c1);
    if (c2) atomicAdd(&hist[2 * KS_BINS + bin], c2);
  };
  auto hist_get = [&](int bin) -> unsigned long long {
    return (unsigned long long)hist[bin] + ((unsigned long long)hist[KS_BINS + bin] << 14) +
           ((unsigned long long)hist[2 * KS_BINS + bin] << 28);
  };

  const int u = blockIdx.x;
  const int r = u % n_req, o = u / n_req;
  const int base = tok_indptr[r];
  const int L = tok_indptr[r + 1] - base;
  int n_keep = 0;
  if (FUSED) {
    n_keep = min(max(fs.budget[r], 0), L);
    // as actkv_select: nothing after an earlier error of the step, and no store past the index buffer
    if (status_set(fs.status)) return;
    if ((int64_t)fs.keep_indptr[r] + n_keep > fs.sel_stride) {
      if (threadIdx.x == 0) report(fs.status, ACTKV_E_INVALID, r, n_keep);
      return;
    }
    if (n_keep == 0 && fs.tie != nullptr && threadIdx.x == 0) fs.tie[u] = actkv_tie_t{0.f, 0, 0, 0};
  }
  if (L <= 0) return;
  float* sc = score + (int64_t)o * sum_tok + base;
  float* ks = keep_score + (int64_t)o * sum_tok + base;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // (two bodies: as a branch inside one, the distinction cost 670 -> 680 us at the end of an action region)
  auto unit = [&](auto is_resident) {
    constexpr bool resident = decltype(is_resident)::value;
    auto key_at = [&](int i) -> uint32_t { return resident ? skeys[i] : order_key(sc[i]); };

    // ---- one read of the scores: order keys into shared memory, their range, the total mass ----
    uint32_t lo = 0xffffffffu, hi = 0u;
    unsigned long long total = 0ull;
    for (int i0 = tid; i0 < L; i0 += 4 * NT) {             // four loads in flight per thread
      float x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) x[j] = i0 + j * NT < L ? sc[i0 + j * NT] : 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (i0 + j * NT < L) {
          const uint32_t k = order_key(x[j]);
          if constexpr (resident) skeys[i0 + j * NT] = k;
          lo = min(lo, k);
          hi = max(hi, k);
          total += ks_mass(x[j]);
        }
      }
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) total += __shfl_xor_sync(0xffffffffu, total, d);
    if (lane == 0) sh.warp_tot[warp] = total;
    block_range<NT>(sh.sel, lo, hi);                       // (its barrier also covers the keys and warp_tot)
    total = lane < WARPS ? sh.warp_tot[lane] : 0ull;
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) total += __shfl_xor_sync(0xffffffffu, total, d);
    // mark = ceil(p_q * total / 10000); total < 2^57 for up to 2^16 entries and p_q <= 10000 < 2^14: the product is
    // taken in two halves to stay inside 64 bits
    const unsigned long long mark = total / 10000ull * (unsigned long long)p_q +
                                    (total % 10000ull * (unsigned long long)p_q + 9999ull) / 10000ull;

    // ---- the largest key T with mass(key >= T) >= mark ----
    uint32_t thr = 0u;                   // key of the last hit
    int32_t last_tie = -1;               // entries equal to it are hits up to this index
    if (mark > 0ull) {                   // (uniform over the CTA)
      unsigned long long above = 0ull;   // mass of keys above the range in question
      uint32_t span = hi - lo;
      for (;;) {
        const int shift = bin_shift(span, KS_BINS);
        for (int i = tid; i < 3 * KS_BINS; i += NT) hist[i] = 0u;
        if (tid == 0) sh.sel.n_list = 0u;
        __syncthreads();
        for (int i = tid; i < L; i += NT) {
          const uint32_t k = key_at(i);
          if (k - lo <= span) hist_add((k - lo) >> shift, ks_mass(key_to_float(k)));
        }
        __syncthreads();
        // sums over the bins, descending
        const int b0 = KS_BINS - PER * (tid + 1);
        unsigned long long h[PER], mine = 0ull;
#pragma unroll
        for (int j = 0; j < PER; ++j) { h[j] = hist_get(b0 + j); mine += h[j]; }
        unsigned long long acc = above + block_exclusive<NT, unsigned long long>(mine, sh.warp_tot);
        if (acc < mark && acc + mine >= mark) {            // exactly one thread
#pragma unroll
          for (int j = PER - 1; j >= 0; --j) {
            if (acc < mark && acc + h[j] >= mark) {
              sh.bin = (uint32_t)(b0 + j);
              sh.above = acc;
            }
            acc += h[j];
          }
        }
        __syncthreads();
        above = sh.above;
        lo += sh.bin << shift;
        span = (1u << shift) - 1u;
        for (int i = tid; i < L; i += NT) {
          const uint32_t k = key_at(i);
          if (k - lo <= span) {
            const uint32_t p = atomicAdd(&sh.sel.n_list, 1u);
            if (p < (uint32_t)KS_LIST) { sh.list[p] = k; sh.mass[p] = ks_mass(key_to_float(k)); }
          }
        }
        __syncthreads();
        const uint32_t count = sh.sel.n_list;
        if (shift == 0) {                                  // a bin is one key
          if (tid == 0) { sh.thr = lo; sh.eq_total = count; }
          break;
        }
        if (count <= (uint32_t)KS_LIST) {
          for (uint32_t i = tid; i < count; i += NT) {
            const uint32_t v = sh.list[i];
            const unsigned long long m = sh.mass[i];
            unsigned long long gt = above;
            uint32_t equal = 0u;
            for (uint32_t j = 0; j < count; ++j) {
              const uint32_t w = sh.list[j];
              gt += w > v ? sh.mass[j] : 0ull;
              equal += w == v;
            }
            if (gt < mark && gt + m * equal >= mark) {     // (every entry of that value: the same words)
              sh.thr = v;
              sh.above = gt;
              sh.eq_total = equal;
            }
          }
          break;
        }
        __syncthreads();
      }
      __syncthreads();
      thr = sh.thr;
      // all entries with key == thr share one score, hence one mass (> 0: the bin crossed the mark)
      const unsigned long long thr_mass = ks_mass(key_to_float(thr));
      const unsigned long long need = mark - sh.above;     // > 0 by construction
      const unsigned long long ties_hit = thr_mass > 0ull ? (need + thr_mass - 1ull) / thr_mass : 0ull;
      last_tie = L;
      if (ties_hit < sh.eq_total) {
        // the index of the ties_hit-th entry equal to thr: a contiguous segment per warp
        const int seg = ((L + WARPS - 1) / WARPS + 31) & ~31;
        const int i_begin = warp * seg, i_end = min(L, i_begin + seg);
        uint32_t n_eq = 0u;
        for (int i = i_begin + lane; i < i_end; i += 32) n_eq += key_at(i) == thr;
        n_eq = __reduce_add_sync(0xffffffffu, n_eq);
        if (lane == 0) sh.sel.warp_eq[warp] = n_eq;
        if (tid == 0) sh.last_tie = -1;
        __syncthreads();
        uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp && lane < WARPS ? sh.sel.warp_eq[lane] : 0u);
        if (ties_hit > before && ties_hit <= before + n_eq) {
          for (int i0 = i_begin; i0 < i_end; i0 += 32) {
            const int i = i0 + lane;
            const bool eq = i < i_end && key_at(i) == thr;
            const uint32_t bal = __ballot_sync(0xffffffffu, eq);
            if (eq && before + __popc(bal & ((2u << lane) - 1u)) == ties_hit) sh.last_tie = i;
            before += __popc(bal);
          }
        }
        __syncthreads();
        last_tie = sh.last_tie;
      }
    }

    // ---- hits, keep-score update, ranking keys: every entry on its own ----
    const int np = n_protect ? n_protect[r] : 0;
    uint32_t* mrow = hit_mask ? hit_mask + (int64_t)o * ((sum_tok + 31) / 32) : nullptr;
    // (the protected entries, which rank as +inf, are counted apart: the range that TopK divides is that of the others)
    constexpr uint32_t INF_KEY = 0xff800000u;
    uint32_t n_inf = 0u;
    lo = 0xffffffffu;
    hi = 0u;
    for (int i0 = tid; i0 < L; i0 += 4 * NT) {
      float old[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) old[j] = i0 + j * NT < L ? ks[i0 + j * NT] : 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int i = i0 + j * NT;
        if (i >= L) break;
        const uint32_t k = key_at(i);
        const bool hit = mark > 0ull && (k > thr || (k == thr && i <= last_tie));
        const float decayed = mul_ieee(lambda, old[j]);
        const float nk = hit ? add_ieee(decayed, key_to_float(k)) : decayed;
        ks[i] = nk;
        const float rank = (i < np) ? INFINITY : nk;            // what TopK ranks
        if (FUSED) {
          const uint32_t rk = order_key(rank);
          if constexpr (resident) skeys[i] = rk;
          if (rk == INF_KEY) {
            ++n_inf;
          } else {
            lo = min(lo, rk);
            hi = max(hi, rk);
          }
        } else {
          sc[i] = rank;
        }
        if (hit && mrow) atomicOr(&mrow[(base + i) >> 5], 1u << ((base + i) & 31));
      }
    }
    if (FUSED && n_keep > 0) {                             // uniform over the CTA
      n_inf = __reduce_add_sync(0xffffffffu, n_inf);
      __syncthreads();                                     // (the ranges of the first block_range have been read)
      if (lane == 0) sh.sel.warp_eq[warp] = n_inf;
      block_range<NT>(sh.sel, lo, hi);
      n_inf = __reduce_add_sync(0xffffffffu, lane < WARPS ? sh.sel.warp_eq[lane] : 0u);
      if (hi > INF_KEY) {                                  // (keys beyond +inf: NaN scores)
        lo = min(lo, INF_KEY);
        n_inf = 0u;
      } else if (n_inf >= (uint32_t)n_keep) {
        lo = hi = INF_KEY;
        n_inf = 0u;
      }
      int32_t* out = fs.sel_idx + (int64_t)o * fs.sel_stride + fs.keep_indptr[r];
      uint32_t* keep_row = fs.keep_mask ? fs.keep_mask + (int64_t)o * ((sum_tok + 31) / 32) : nullptr;
      if constexpr (resident)
        select_and_emit<NT, KS_BINS>([&](int i) { return skeys[i]; }, hist, sh.sel, lo, hi, L, n_keep, out, keep_row, base, fs.tie, u,
                                     (int)n_inf);
      else
        select_and_emit<NT, KS_BINS>([&](int i) { return order_key(i < np ? INFINITY : ks[i]); }, hist, sh.sel, lo, hi, L, n_keep, out,
                                     keep_row, base, fs.tie, u, (int)n_inf);
    }
  };
  if (L <= cap) unit(std::true_type{}); else unit(std::false_type{});      // (uniform over the CTA)
}

// max_tok: a bound on the unit lengths.
template <bool FUSED, int NT>
static int keepscore_launch_n(float* score, const int32_t* tok_indptr, int32_t sum_tok, int32_t max_tok, int64_t units,
                              int32_t n_req, int32_t p_q, float lambda, const int32_t* n_protect, float* keep_score,
                              uint32_t* hit_mask, const FusedSelectArgs& fs, cudaStream_t s) {
  constexpr size_t fixed = 3 * KS_BINS * 4;
  const size_t smem = resident_smem(fixed, max_tok);
  if (ensure_dyn_smem(keepscore_kernel<FUSED, NT>, smem) != cudaSuccess) return ACTKV_E_CUDA;
  launch_pdl(keepscore_kernel<FUSED, NT>, (unsigned)units, NT, smem, s, score, tok_indptr, sum_tok, n_req, p_q, lambda,
             n_protect, keep_score, hit_mask, (int32_t)((smem - fixed) / 4), fs);
  ACTKV_CHECK_LAUNCH();
  return ACTKV_OK;
}
template <bool FUSED>
static int keepscore_launch(float* score, const int32_t* tok_indptr, int32_t sum_tok, int32_t max_tok, int64_t units, int32_t n_req,
                            int32_t p_q, float lambda, const int32_t* n_protect, float* keep_score, uint32_t* hit_mask,
                            const FusedSelectArgs& fs, cudaStream_t s) {
  const int nt = select_threads(units, max_tok);
  if (nt == 256)
    return keepscore_launch_n<FUSED, 256>(score, tok_indptr, sum_tok, max_tok, units, n_req, p_q, lambda, n_protect, keep_score,
                                          hit_mask, fs, s);
  if (nt == 512)
    return keepscore_launch_n<FUSED, 512>(score, tok_indptr, sum_tok, max_tok, units, n_req, p_q, lambda, n_protect, keep_score,
                                          hit_mask, fs, s);
  return keepscore_launch_n<FUSED, 1024>(score, tok_indptr, sum_tok, max_tok, units, n_req, p_q, lambda, n_protect, keep_score,
                                         hit_mask, fs, s);
}

constexpr int GA_NT = 256, GA_PER = 4;
// GA_PER survivors per thread, all loads of one kind in flight together; the request is searched once per CTA (by every
// warp, 32 offsets at a time) and, where the CTA's survivors belong to several, advanced from there.  64 rows of 197 K survivors 68.8 -> 31.3 us (4.8 TB/s; two per thread 39.5, eight 30.6).
__global__ void __launch_bounds__(GA_NT) gather_f32_kernel(
    const float* __restrict__ src, int64_t src_stride, const int32_t* __restrict__ tok_indptr,
    const int32_t* __restrict__ sel_idx, int64_t sel_stride, const int32_t* __restrict__ keep_indptr, int32_t n_req,
    float* __restrict__ dst, int64_t dst_stride) {
  pdl_begin(src, tok_indptr, sel_idx, keep_indptr);
  const int o = blockIdx.y, lane = threadIdx.x & 31;
  const int32_t* sel = sel_idx + (int64_t)o * sel_stride;
  const float* sc = src + (int64_t)o * src_stride;
  float* out = dst + (int64_t)o * dst_stride;
  const int total = keep_indptr[n_req];
  // (one round when the host's bound holds)
  for (int64_t first64 = (int64_t)blockIdx.x * (GA_NT * GA_PER); first64 < total; first64 += (int64_t)gridDim.x * (GA_NT * GA_PER)) {
    const int first = (int)first64, i0 = first + threadIdx.x;
    int tok[GA_PER];
#pragma unroll
    for (int k = 0; k < GA_PER; ++k) tok[k] = i0 + k * GA_NT < total ? sel[i0 + k * GA_NT] : 0;
    // the request of the CTA's first survivor: the last r with keep_indptr[r] <= first
    int r = 0;
    for (int q0 = 1; q0 < n_req; q0 += 32) {
      const int c = __popc(__ballot_sync(0xffffffffu, q0 + lane < n_req && keep_indptr[q0 + lane] <= first));
      r += c;
      if (c < 32) break;
    }
    int next = keep_indptr[r + 1], base = tok_indptr[r];
    if (next >= min(total, first + GA_NT * GA_PER)) {          // one request (uniform over the CTA)
      float v[GA_PER];
#pragma unroll
      for (int k = 0; k < GA_PER; ++k) v[k] = i0 + k * GA_NT < total ? sc[base + tok[k]] : 0.f;
#pragma unroll
      for (int k = 0; k < GA_PER; ++k)
        if (i0 + k * GA_NT < total) out[i0 + k * GA_NT] = v[k];
    } else {
#pragma unroll
      for (int k = 0; k < GA_PER; ++k) {
        const int i = i0 + k * GA_NT;
        if (i < total) {
          while (i >= next) {                                  // (i < total = keep_indptr[n_req]: r + 1 < n_req here)
            ++r;
            next = keep_indptr[r + 1];
            base = tok_indptr[r];
          }
          out[i] = sc[base + tok[k]];
        }
      }
    }
  }
}

}  // namespace actkv

// longest unit of the one-launch form (the header names the figure)
constexpr int32_t KS_FUSED_MAX = 45568;
static_assert(3 * actkv::KS_BINS * 4 + (size_t)KS_FUSED_MAX * 4 <= actkv::SEL_SMEM_MAX, "fits in shared memory");

extern "C" {

int actkv_keepscore(float* score, const int32_t* tok_indptr, int32_t sum_tok, int32_t n_outer, int32_t n_req,
                    float top_p, float lambda, const int32_t* n_protect, float* keep_score, uint32_t* hit_mask,
                    int32_t* status, actkv_stream_t stream) {
  (void)status;
  if (n_outer < 0 || n_req < 0 || sum_tok < 0) return ACTKV_E_INVALID;
  if (!(top_p >= 0.f && top_p <= 1.f) || !(lambda >= 0.f && lambda <= 1.f)) return ACTKV_E_INVALID;
  if (n_outer == 0 || n_req == 0 || sum_tok == 0) return ACTKV_OK;
  if (!score || !tok_indptr || !keep_score) return ACTKV_E_INVALID;
  const int64_t units = (int64_t)n_outer * n_req;
  if (units > 0x7fffffffLL) return ACTKV_E_INVALID;
  const int32_t p_q = (int32_t)lrintf(top_p * 10000.f);
  // (no unit is longer than all of them together)
  return actkv::keepscore_launch<false>(score, tok_indptr, sum_tok, sum_tok, units, n_req, p_q, lambda, n_protect, keep_score,
                                        hit_mask, actkv::FusedSelectArgs{}, (cudaStream_t)stream);
}

int actkv_keepscore_select(float* score, const int32_t* tok_indptr, int32_t sum_tok, int32_t max_tok, int32_t n_outer,
                           int32_t n_req, float top_p, float lambda, const int32_t* n_protect, float* keep_score,
                           uint32_t* hit_mask, const int32_t* budget, const int32_t* keep_indptr, int32_t* sel_idx,
                           int64_t sel_stride, uint32_t* keep_mask, actkv_tie_t* tie_report, int32_t* status,
                           actkv_stream_t stream) {
  if (n_outer < 0 || n_req < 0 || sum_tok < 0 || max_tok < 0 || sel_stride < 0) return ACTKV_E_INVALID;
  if (!(top_p >= 0.f && top_p <= 1.f) || !(lambda >= 0.f && lambda <= 1.f)) return ACTKV_E_INVALID;
  if (n_outer == 0 || n_req == 0 || sum_tok == 0) return ACTKV_OK;
  if (!score || !tok_indptr || !keep_score || !budget || !keep_indptr || !sel_idx) return ACTKV_E_INVALID;
  if (max_tok > KS_FUSED_MAX) {
    // a unit that does not fit in shared memory: the two stages as two kernels (the ranking keys go through `score`)
    int rc = actkv_keepscore(score, tok_indptr, sum_tok, n_outer, n_req, top_p, lambda, n_protect, keep_score, hit_mask,
                             status, stream);
    if (rc != ACTKV_OK) return rc;
    return actkv_select(score, tok_indptr, sum_tok, budget, n_outer, n_req, keep_indptr, sel_idx, sel_stride, keep_mask,
                        tie_report, nullptr, 0, status, stream);
  }
  const int64_t units = (int64_t)n_outer * n_req;
  if (units > 0x7fffffffLL) return ACTKV_E_INVALID;
  const int32_t p_q = (int32_t)lrintf(top_p * 10000.f);
  actkv::FusedSelectArgs fs{budget, keep_indptr, sel_idx, sel_stride, keep_mask, tie_report, status};
  return actkv::keepscore_launch<true>(score, tok_indptr, sum_tok, max_tok, units, n_req, p_q, lambda, n_protect, keep_score,
                                       hit_mask, fs, (cudaStream_t)stream);
}

int actkv_gather_f32(const float* src, int64_t src_stride, const int32_t* tok_indptr, const int32_t* sel_idx,
                     int64_t sel_stride, const int32_t* keep_indptr, int32_t n_outer, int32_t n_req,
                     int32_t max_total_keep, float* dst, int64_t dst_stride, actkv_stream_t stream) {
  if (n_outer < 0 || n_req < 0 || max_total_keep < 0) return ACTKV_E_INVALID;
  if (n_outer == 0 || n_req == 0 || max_total_keep == 0) return ACTKV_OK;
  if (!src || !tok_indptr || !sel_idx || !keep_indptr || !dst || n_outer > 65535) return ACTKV_E_INVALID;
  const dim3 grid((unsigned)((max_total_keep + actkv::GA_NT * actkv::GA_PER - 1) / (actkv::GA_NT * actkv::GA_PER)), (unsigned)n_outer);
  actkv::launch_pdl(actkv::gather_f32_kernel, grid, actkv::GA_NT, 0, (cudaStream_t)stream, src, src_stride, tok_indptr,
                    sel_idx, sel_stride, keep_indptr, n_req, dst, dst_stride);
  ACTKV_CHECK_LAUNCH();
  return ACTKV_OK;
}

}  // extern "C"
