// actkv_select: TopK(score, k = B) per (layer x KV head, request) unit — Algorithm 1, step 5,
// applied to the pooled action-region score.  One CTA per unit.  The unit's scores are read once and
// kept in shared memory as order-preserving 32-bit keys (up to 52 K tokens; longer units re-read them
// from L2); select_core.cuh finds the n-th largest key exactly and emits the kept indices.
//
// What bounds it: latency.  A unit is four sweeps over shared memory between a dozen barriers, so short units run with
// small CTAs and only the shared memory that the host's bound on the lengths asks for, several per SM.
// 512 units of 35000 keys 104 -> 83 us, 1024 of 16000 115 -> 82, 2048 of 1500 90 -> 34, 8 of 4096 9.7 -> 8.7 (fixed
// digits of 12, 12 and 8 bits and an emitting sweep with block scans before).
#include "select_core.cuh"

namespace actkv {

template <int NT, int BINS>
__global__ void __launch_bounds__(NT) select_kernel(
    const float* __restrict__ score, const int32_t* __restrict__ tok_indptr, int32_t sum_tok,
    const int32_t* __restrict__ budget, int32_t n_req, const int32_t* __restrict__ keep_indptr,
    int32_t* __restrict__ sel_idx, int64_t sel_stride, uint32_t* __restrict__ keep_mask,
    actkv_tie_t* __restrict__ tie, int32_t cap, int32_t* status) {
  pdl_begin(score, tok_indptr, budget, keep_indptr);
  extern __shared__ __align__(16) uint32_t sel_smem[];
  __shared__ SelectShared<NT> sh;
  uint32_t* hist = sel_smem;                             // [BINS]
  uint32_t* skeys = sel_smem + BINS;                     // [cap]
  const int u = blockIdx.x;
  const int r = u % n_req, o = u / n_req;
  const int base = tok_indptr[r], end = tok_indptr[r + 1], b_raw = budget[r], kept = keep_indptr[r];
  const int L = end - base;
  const int n = min(b_raw < 0 ? 0 : b_raw, L);
  const float* sc = score + (int64_t)o * sum_tok + base;
  const int tid = threadIdx.x;

  // An earlier stage of the step failed (a score kernel that gave up, a bad table): its scores are not
  // consumed.  A budget the host did not size the index buffer for (the budgets are device data, e.g.
  // straight from actkv_budget) is reported before anything is stored.
  if (status_set(status)) return;
  if ((int64_t)kept + n > sel_stride) {
    if (tid == 0) report(status, ACTKV_E_INVALID, r, n);
    return;
  }
  if (n == 0) {
    if (tie != nullptr && tid == 0) tie[u] = actkv_tie_t{0.f, 0, 0, 0};
    return;
  }
  const bool resident = L <= cap;                        // uniform over the CTA
  uint32_t lo = 0xffffffffu, hi = 0u;
  // The one read of the scores (16-byte vectors between an unaligned head and tail) also takes their range.
  {
    auto take = [&](int i, float x) {
      const uint32_t k = order_key(x);
      if (resident) skeys[i] = k;
      lo = min(lo, k);
      hi = max(hi, k);
    };
    const int head = min(L, (int)((16u - ((uint32_t)(uintptr_t)sc & 15u)) & 15u) >> 2);
    const int n_vec = (L - head) >> 2;
    if (tid < head) take(tid, sc[tid]);
    const float4* sc4 = reinterpret_cast<const float4*>(sc + head);
    // (four loads in flight per thread: the read is bound by latency, not by bandwidth)
    for (int v0 = tid; v0 < n_vec; v0 += 4 * NT) {
      float4 x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int v = v0 + j * NT;
        x[j] = v < n_vec ? __ldg(sc4 + v) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int v = v0 + j * NT;
        if (v < n_vec) {
          const int i = head + 4 * v;
          take(i, x[j].x); take(i + 1, x[j].y); take(i + 2, x[j].z); take(i + 3, x[j].w);
        }
      }
    }
    const int tail0 = head + 4 * n_vec;
    if (tail0 + tid < L) take(tail0 + tid, sc[tail0 + tid]);
  }
  block_range<NT>(sh, lo, hi);
  int32_t* out = sel_idx + (int64_t)o * sel_stride + kept;
  uint32_t* mask_row = keep_mask ? keep_mask + (int64_t)o * ((sum_tok + 31) / 32) : nullptr;
  if (resident)
    select_and_emit<NT, BINS>([&](int i) { return skeys[i]; }, hist, sh, lo, hi, L, n, out, mask_row, base, tie, u);
  else
    select_and_emit<NT, BINS>([&](int i) { return order_key(sc[i]); }, hist, sh, lo, hi, L, n, out, mask_row, base, tie, u);
}

template <int NT, int BINS>
static int select_launch_n(const float* score, const int32_t* tok_indptr, int32_t sum_tok, int32_t max_tok, const int32_t* budget,
                           int64_t units, int32_t n_req, const int32_t* keep_indptr, int32_t* sel_idx, int64_t sel_stride,
                           uint32_t* keep_mask, actkv_tie_t* tie_report, int32_t* status, cudaStream_t s) {
  const size_t smem = resident_smem(BINS * 4, max_tok);
  if (ensure_dyn_smem(select_kernel<NT, BINS>, smem) != cudaSuccess) return ACTKV_E_CUDA;
  launch_pdl(select_kernel<NT, BINS>, (unsigned)units, NT, smem, s, score, tok_indptr, sum_tok, budget, n_req, keep_indptr,
             sel_idx, sel_stride, keep_mask, tie_report, (int32_t)((smem - BINS * 4) / 4), status);
  ACTKV_CHECK_LAUNCH();
  return ACTKV_OK;
}

int select_launch(const float* score, const int32_t* tok_indptr, int32_t sum_tok, int32_t max_tok, const int32_t* budget,
                  int32_t n_outer, int32_t n_req, const int32_t* keep_indptr, int32_t* sel_idx, int64_t sel_stride,
                  uint32_t* keep_mask, actkv_tie_t* tie_report, int32_t* status, cudaStream_t stream) {
  if (n_outer < 0 || n_req < 0 || sum_tok < 0 || sel_stride < 0) return ACTKV_E_INVALID;
  if (n_outer == 0 || n_req == 0) return ACTKV_OK;
  if (!score || !tok_indptr || !budget || !keep_indptr || !sel_idx) return ACTKV_E_INVALID;
  const int64_t units = (int64_t)n_outer * n_req;
  if (units > 0x7fffffffLL) return ACTKV_E_INVALID;
  const int nt = select_threads(units, max_tok);
  if (nt == 256)
    return select_launch_n<256, 2048>(score, tok_indptr, sum_tok, max_tok, budget, units, n_req, keep_indptr, sel_idx,
                                      sel_stride, keep_mask, tie_report, status, stream);
  if (nt == 512)
    return select_launch_n<512, 4096>(score, tok_indptr, sum_tok, max_tok, budget, units, n_req, keep_indptr, sel_idx,
                                      sel_stride, keep_mask, tie_report, status, stream);
  return select_launch_n<1024, 4096>(score, tok_indptr, sum_tok, max_tok, budget, units, n_req, keep_indptr, sel_idx,
                                     sel_stride, keep_mask, tie_report, status, stream);
}

// One warp: inclusive scans of 32 requests at a time.
__global__ void keep_indptr_kernel(const int32_t* seq_len, const int32_t* budget, int32_t n_req, int32_t* keep_indptr) {
  pdl_begin();
  const int lane = threadIdx.x;
  int32_t acc = 0;
  if (lane == 0) keep_indptr[0] = 0;
  for (int r0 = 0; r0 < n_req; r0 += 32) {
    const int r = r0 + lane;
    int32_t v = r < n_req ? min(max(budget[r], 0), seq_len[r]) : 0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int32_t t = __shfl_up_sync(0xffffffffu, v, d);
      if (lane >= d) v += t;
    }
    if (r < n_req) keep_indptr[r + 1] = acc + v;
    acc += __shfl_sync(0xffffffffu, v, 31);
  }
}

}  // namespace actkv

extern "C" {

size_t actkv_select_workspace_bytes(int32_t, int32_t, int32_t) { return 0; }

int actkv_select(const float* score, const int32_t* tok_indptr, int32_t sum_tok,
                 const int32_t* budget, int32_t n_outer, int32_t n_req,
                 const int32_t* keep_indptr, int32_t* sel_idx, int64_t sel_stride,
                 uint32_t* keep_mask, actkv_tie_t* tie_report, void* ws, size_t ws_bytes,
                 int32_t* status, actkv_stream_t stream) {
  (void)ws; (void)ws_bytes;
  // (no unit is longer than all of them together)
  return actkv::select_launch(score, tok_indptr, sum_tok, sum_tok, budget, n_outer, n_req, keep_indptr, sel_idx, sel_stride,
                              keep_mask, tie_report, status, (cudaStream_t)stream);
}

int actkv_keep_indptr(const int32_t* seq_len, const int32_t* budget, int32_t n_req,
                      int32_t* keep_indptr, actkv_stream_t stream) {
  if (n_req < 0 || !keep_indptr || (n_req > 0 && (!seq_len || !budget))) return ACTKV_E_INVALID;
  actkv::launch_pdl(actkv::keep_indptr_kernel, 1, 32, 0, (cudaStream_t)stream, seq_len, budget, n_req, keep_indptr);
  ACTKV_CHECK_LAUNCH();
  return ACTKV_OK;
}

}  // extern "C"
