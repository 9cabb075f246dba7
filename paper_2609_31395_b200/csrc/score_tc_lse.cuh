// LSE pass of the tensor-core score path (Section 7.1, LSE equation):
//   lse[row] = log sum_{key visible} exp(sm_scale * q_row . k_key),   row = (window token w, group head g).
//
// D[row, key] = Q K^T with the rows on the TMEM lanes, so every epilogue thread owns one row per
// 128-row block and folds its share of the row's logits into a running (reference, sum of exp2): no
// shuffles.  A work item is up to three row blocks of a unit (two where a window is longer than 384 rows) x one chunk of keys; the items of
// a longer window stand side by side and each fetches the keys.
//
// Operand placement.  An A operand in shared memory is re-read for every MMA and that read is not
// overlapped with the MMA (measured 105 cycles per 128x128x16 MMA against 74 with A in tensor memory,
// 64 nominal).  The Q blocks are the same for every key tile of the item, so they are copied once into
// tensor memory and used as the A operand from there; only the K tile (B) streams through shared memory.
// TMEM columns: [0,256) Q blocks, [256,512) two 128-column accumulators; a job is one
// (key tile, row block) product.  Even jobs go to accumulator 0, odd jobs to accumulator 1; each
// accumulator has its own MMA-issuing warp and its own group of eight epilogue warps (64 columns per
// thread), which hand the accumulator back as soon as their columns are in registers.  While one group
// waits for tensor memory the other keeps the special function unit busy.
//
// Items.  One CTA per SM, which goes on from item to item: the first is its own blockIdx, the next ones those of CTAs that have
// not been launched yet (cluster launch control), so requests of different lengths and windows spread over the SMs by themselves.
// In the ring of stages an item is its Q blocks, then its K tiles; the producers run ahead into the next item, whose
// Q blocks go to the other half of the Q columns (three blocks at head_dim 128 wait for it), and warp 3 merges the shares of an item while
// the epilogue is in the next.  With a CTA per item 12 to 20 K cycles passed before its first job was done, beside 1030 for a job; from item to item it is 2 K.  With one
// producer a unit of one row block waited for its key tiles.  A last block of at most 64 rows is held twice and each copy folds half of
// its columns.
// LSE pass, us, before and after: 4 layers x 8 heads, 8 x 16000 keys, 128 rows 280 -> 184, 192 rows 332 -> 284, head_dim 64 and 256 rows
// 309 -> 289; 2 x 32768 keys, 256 rows 190 -> 170; 4 x 16000 keys, 512 rows 320 -> 301; 8 layers x 8 heads, 16 requests of
// 12000-20000 keys and 140-348 rows 1628 -> 1387.  In a loop of seconds, at the power cap: 36 layers of 32768 keys, 256 rows 828 -> 823, 8 layers of
// 8 x 35000 keys, 512 rows 1440 -> 1420.  Slower than a CTA per unit: 353 to 384 rows (4 x 16000 keys, 384 rows 240 -> 252; with two items a
// unit 258).
//
// What bounds the kernel (measured on B200 with micro-benchmarks and per-job timestamps):
//  * Issuing is not free: a tcgen05.mma costs the issuing thread about 50 cycles and a tcgen05.commit
//    about 80, some 470 cycles for a job the tensor pipe executes in 512, and the commit reaches the
//    waiting warps about 240 cycles after the last MMA retires; hence two issuers.
//  * An SM sub-partition dispatches about one fp32 operation per clock (the packed fp32x2 forms take
//    two, so they save nothing) and its special function unit delivers one warp-wide exp2 per 8 clocks.
//    One exp2 per (row, key) on that unit alone costs 8 clocks per warp and logit against 4.6 for the
//    contraction: the pass is bound by the exp rate.  Of each 8 columns, NPOLY take a polynomial on the
//    FMA pipe instead (ten dispatch slots each, against three slots and eight clocks of the unit); the
//    two kinds overlap only partly, and NPOLY = 1 measured best (16 layers of 8 x 35000 keys, 512 rows:
//    0: 2.83 ms, 1: 2.75, 2: 2.84).
//  * To keep the slot count low there is no running maximum: the reference e of a row is the maximum of
//    the first logits the thread saw, in log2 units and rounded to an integer; later logits may exceed it
//    (2^x is evaluated for x up to 126), and only if a partial sum grows past 2^40 is the reference moved (a
//    rare, slower path that also serves tiles cut by the end of the request or by the causal diagonal).
// Polynomial: textbook range reduction (Cody and Waite, Software Manual for the Elementary Functions, 1980):
// x = v c = j + f with j the nearest integer (adding and subtracting 1.5 2^23) and f in [-0.5, 0.5], 2^f by a cubic
// fitted here (max relative error 7.5e-5, far inside the 2e-3 score tolerance), 2^(j - e) from an exponent field,
// j - e clamped to [-126, 126].  The reference being an integer, it enters in that factor only.
#pragma once

#include "tc_common.cuh"

namespace actkv {
namespace tc {

constexpr int LSE_NPOLY = 1;                     // columns of every 8 whose exp2 is the polynomial
constexpr float EXP2_ROUND = 12582912.f;         // 1.5 * 2^23: adding it rounds to the nearest integer

// The cubic's coefficients come with the kernel's parameters, as operands from the constant bank: as literals they are brought in by
// instructions of their own (2 x 32768 keys, 256 rows: 176.5 us against 173.6; from a __constant__ array 175).
constexpr float EXP2_C0 = 0.9999280571937561f, EXP2_C1 = 0.6932609677314758f, EXP2_C2 = 0.2426111251115799f, EXP2_C3 = 0.0551716648042202f;

// 2^(v c - e) for an integer e; base = EXP2_ROUND + 127 - e.  2^(j - e) is multiplied in, not added to the exponent field of p:
// beyond |v c| = 2^22, where f leaves its interval, and for infinite and NaN logits the product is then as small as it has to be,
// or larger than LSE_BIG, or NaN, and the caller takes the general form.
__device__ __forceinline__ float exp2_poly(float v, float c, float base, const Exp2Cubic& k) {
  const float t = fmaf(v, c, base);                                // j - e + 127, j = round(v c): the exponent field, in the low bits
  const float f = fmaf(v, c, base - t);                            // v c - j
  float p = fmaf(k.c3, f, k.c2);
  p = fmaf(p, f, k.c1);
  p = fmaf(p, f, k.c0);
  const float e = fminf(fmaxf(t, EXP2_ROUND + 1.f), EXP2_ROUND + 253.f);
  return p * __int_as_float(__float_as_int(e) << 23);
}

// 32 logits of one row, all visible, against the row's reference e (finite, below LSE_REF_MAX): returns
// sum_i 2^(v_i c - e).  Two partial sums: the registers that more of them take cost more than the shorter chains give
// (2.75 ms with two, 2.86 with four, for 16 layers of 8 x 35000 keys and 512 rows).
template <int NPOLY>
__device__ __forceinline__ float lse_fast32(const float* v, float c, float neg_e, const Exp2Cubic& k) {
  float s[2] = {0.f, 0.f};
  const float base = EXP2_ROUND + 127.f + neg_e;
#pragma unroll
  for (int g8 = 0; g8 < 4; ++g8) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float x = v[g8 * 8 + i];
      // the polynomial columns are spread over the group so that the two kinds interleave in program order
      const bool poly = (NPOLY >= 1 && i == 4) || (NPOLY >= 2 && i == 1) || (NPOLY >= 3 && i == 6) || (NPOLY >= 4 && i == 3);
      s[i & 1] += poly ? exp2_poly(x, c, base, k) : exp2f(fmaf(x, c, neg_e));
    }
  }
  return s[0] + s[1];
}

// The general form: logits n_lo <= i < nv (any integers) are visible; moves the reference to the maximum seen
// so far.  Also the entry for a row's first logits (e = -inf, sum = 0).
__device__ __forceinline__ void lse_slow32(const float* v, int n_lo, int nv, float c, float& e, float& sum) {
  if (nv <= 0 || n_lo >= 32 || n_lo >= nv) return;
  float gm = -INFINITY;
#pragma unroll
  for (int i = 0; i < 32; ++i) gm = fmaxf(gm, (i >= n_lo && i < nv) ? v[i] : -INFINITY);
  const float ge = rintf(gm * c);
  if (ge > e) { sum = (e == -INFINITY) ? 0.f : sum * exp2f(e - ge); e = ge; }
#pragma unroll
  for (int i = 0; i < 32; ++i) sum += (i >= n_lo && i < nv) ? exp2f(fmaf(v[i], c, -e)) : 0.f;
}

constexpr int LSE_EPI_WARPS = 16;                // (TMEM lane quarter, accumulator, column half)
// Warps 0 and 2 are the producers, warps 1 and 3 the MMA issuers, warps 4..19 the epilogue: five warps on each scheduler, which leaves
// a thread up to 102 registers (the epilogue has a use for 96; with a sixth warp it would be 80).
constexpr int LSE_EPI_WARP0 = 4;
constexpr int LSE_THREADS = (LSE_EPI_WARP0 + LSE_EPI_WARPS) * 32;
constexpr int LSE_SLOTS = 2;                     // accumulators
constexpr int LSE_MB = 3;                        // row blocks of an item, at most
constexpr int LSE_A_COLS = 256;                  // TMEM columns holding Q blocks, a half for each of two items
constexpr int LSE_ITEMS_AHEAD = 3;               // item descriptors in shared memory
__host__ __device__ constexpr int lse_stages(int nh) { return nh == 1 ? 8 : 6; }             // K tiles (or Q blocks) in shared memory
constexpr float LSE_BIG = 1099511627776.f;       // 2^40: a partial sum beyond it moves the reference
constexpr float LSE_REF_MAX = 1048576.f;         // references beyond 2^20 (rounding to integers needs |v c| < 2^22) take the general form

// Row groups per unit of a launch whose longest window has `rows` rows, and rows of a group: two blocks, or one group of three.  A third
// block as an item of its own fetches all key tiles once more for half the products (4 layers x 8 heads, 4 x 16000 keys, us, two items / one:
// 260 rows 250 / 219, 320 251 / 223, 384 258 / 252; head_dim 64, 8 layers, 4 x 11000 keys, group 8: 264 rows 300 / 279, 384 326 / 314).  Beyond
// 384 rows groups of three were slower than of two, since fewer and larger items end less evenly: 640 rows, 2 layers x 4 heads, 4 x 8000 keys
// 67.5 / 75.3.
__host__ __device__ constexpr int lse_row_groups(int rows) { return rows <= 384 ? 1 : (rows + 255) / 256; }
__host__ __device__ constexpr int lse_group_rows(int n_rg) { return n_rg == 1 ? 384 : 256; }

// Two blocks of which the second is short change places on odd tiles (exclusive or with this): the short one would otherwise always
// fall to the same accumulator.
__device__ __forceinline__ int lse_flip(int rows) { return (rows + 63) / 64 == 3 ? 1 : 0; }
// Launches whose longest window is an item of blocks that change places with every job (these two, and three): the kernel that keeps
// all (reference, sum) in registers, four more.  384 rows 265 -> 252 us, 192 rows 177 -> 174 (4 layers x 8 heads, 4 x 16000 keys), 16 requests of
// 140-348 rows 1565 -> 1543; other launches are slower with it: 512 rows, 8 x 35000 keys, 1405 -> 1415, a step of one 4K request 38.04 -> 38.27.
inline bool lse_moves(int rows) { return rows > 256 ? rows <= 384 : rows > 128 && rows <= 192; }

// A work item: the rows [row0, row0 + rows) of a unit against n_tiles key tiles.  n_tiles = 0: no more items.
struct LseItem {
  int32_t u, chunk, layer_h, r, L, W, w0, row0, rows, t_begin, n_tiles, slab;
};

struct LseBarriers {
  uint64_t k_full[8];
  uint64_t k_empty[8];
  uint64_t item_full[LSE_ITEMS_AHEAD];
  uint64_t item_empty[LSE_ITEMS_AHEAD];
  uint64_t q_ready[2];          // the Q blocks of an item are in this half of the Q columns
  uint64_t q_free[2];           // the MMAs that read this half of the Q columns have completed
  uint64_t tmem_full[LSE_SLOTS];
  uint64_t tmem_empty[LSE_SLOTS];
  uint64_t shares_full[2];      // the epilogue warps' shares of an item are in `state`
  uint64_t shares_empty[2];     // ... have been merged
  uint64_t clc;
  uint64_t drained[2];
  uint32_t tmem_base;
  int abort_flag;
  uint32_t k_last[8];           // parity of a stage's last load (RING_UNUSED: none yet)
  int at[2];                    // unit and chunk of the item that is being contracted (the first one at first): where a wait gave up
  alignas(16) uint32_t clc_resp[4];
  LseItem item[LSE_ITEMS_AHEAD];
  float2 state[2][2][LSE_MB][2][128];  // (reference e, sum of 2^(v c - e)) per (item parity, group, row block, column half, TMEM lane)
};
static_assert(6 * 2 * HALF_BYTES + sizeof(LseBarriers) <= SMEM_LIMIT, "shared memory");

// After tcgen05.wait::ld: ties the loaded registers to the wait, so that no use of them is scheduled
// ahead of it (the loads are asynchronous; the compiler sees their outputs as defined at issue).
template <int N>
__device__ __forceinline__ void tmem_ld_fence(float* v) {
#pragma unroll
  for (int i = 0; i < N; ++i) asm volatile("" : "+f"(v[i]));
}

// One job as one epilogue warp sees it: the warp takes 64 columns of the accumulator of its group (32 where the block holds its rows
// twice), hands the accumulator back as soon as they are in registers, and folds them into the row's (reference, sum) `ms`.  The two
// groups work on alternate jobs, so while one waits for tensor memory the other keeps the special function unit busy.
//   tq      tensor-memory address of the group's accumulator, this warp's lane quarter and first column
//   wide    64 columns (uniform over the CTA)
//   nv_min  visible columns (from the warp's first column) of the most restricted row of this thread
//   nlo_max columns (from the warp's first column) below the first visible key of the most restricted row
//   last_key()  last visible key of this thread's row; only the slow path needs it and the loop is short of registers
//   key0    key of the warp's first column
// WIN: the layer has a sliding window (a first visible key per row); kept out of the common instantiation, whose
// epilogue should not carry the second bound.
// What is not an exponential counts: an instruction more per job and warp is 0.2 % of the pass, a second unrolled copy of the fold 7 %.
template <int NPOLY, bool WIN, class LastKey>
__device__ __forceinline__ bool lse_job(LseBarriers* bars, volatile int* abort_flag, uint32_t tq, int grp, uint32_t parity, bool wide,
                                        LastKey last_key, float2& ms, int nv_min, int nlo_max, int win_left, int key0, float c,
                                        const Exp2Cubic& cubic, long long wait_cycles) {
  float v[64];
  if (!mbar_wait_warp(smem_u32(&bars->tmem_full[grp]), parity, abort_flag, wait_cycles)) return false;
  tc_fence_after();
  tmem_ld32(tq, v);
  if (wide) tmem_ld32(tq + 32, v + 32);
  tmem_ld_wait();
  tmem_ld_fence<64>(v);
  tc_fence_before();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(smem_u32(&bars->tmem_empty[grp]));
  // (a reference of -inf, before the row's first logits, fails the last test)
  bool slow = __any_sync(0xffffffffu, nv_min < (wide ? 64 : 32) || (WIN && nlo_max > 0) || !(fabsf(ms.x) < LSE_REF_MAX));
  if (!slow) {
    float ps = lse_fast32<NPOLY>(v, c, -ms.x, cubic);
    if (wide) ps += lse_fast32<NPOLY>(v + 32, c, -ms.x, cubic);
    slow = __any_sync(0xffffffffu, !(fabsf(ps) < LSE_BIG));
    if (!slow) ms.y += ps;
  }
  if (slow) {
    const int nv = last_key() - key0 + 1;
    const int nlo = WIN && win_left > 0 ? nv - win_left : 0;
    lse_slow32(v, nlo, nv, c, ms.x, ms.y);
    if (wide) lse_slow32(v + 32, nlo - 32, nv - 32, c, ms.x, ms.y);
  }
  return true;
}

// The item that the CTA with this index stands for; n_tiles <= 0 when there is nothing to contract.  Reports invalid windows, and
// writes the partials of a chunk no row of which sees a key.  Called by a whole warp.
template <bool WIN>
__device__ __forceinline__ LseItem lse_item(const TcArgs& ta, int id, int lane) {
  const ScoreArgs& a = ta.a;
  const int R = a.tab.n_req, Hkv = a.pool.n_kv_heads, G = a.group;
  LseItem x;
  x.n_tiles = 0;
  const int cu = id / ta.n_rg, rg = id - cu * ta.n_rg;   // row group
  x.u = cu / a.n_chunks;
  x.chunk = cu - x.u * a.n_chunks;
  x.r = x.u % R;
  const int h = (x.u / R) % Hkv;
  x.slab = x.u / (R * Hkv);
  x.layer_h = h;
  x.L = a.tab.seq_len[x.r];
  x.w0 = a.win_indptr[x.r];
  x.W = a.win_indptr[x.r + 1] - x.w0;
  x.row0 = rg * lse_group_rows(ta.n_rg);
  x.rows = min(x.W * G - x.row0, lse_group_rows(ta.n_rg));
  const int key_begin = x.chunk * a.lse_chunk;
  if (key_begin >= x.L || (rg > 0 && x.rows <= 0)) return x;
  if (x.W <= 0 || (a.causal && x.W > x.L)) {
    if (lane == 0 && x.chunk == 0 && rg == 0) report(a.status, ACTKV_E_INVALID, x.r, x.W);
    return x;
  }
  // the host sized the grid and the partials from upper bounds of the window and the length
  if (x.W * G > a.rows_max || x.L > a.n_chunks * a.lse_chunk) {
    if (lane == 0 && x.chunk == 0 && rg == 0) report(a.status, ACTKV_E_INVALID, x.r, x.W * G > a.rows_max ? x.W : x.L);
    return x;
  }
  const int t_end = min((x.L + TK - 1) / TK, key_begin / TK + a.lse_chunk / TK);
  // sliding-window layer: key tiles below the first key any row of the unit sees are not fetched at all
  const int lo_all = (WIN && a.win_left > 0) ? max(0, (a.causal ? x.L - x.W : x.L - 1) - a.win_left + 1) : 0;
  x.t_begin = max(key_begin / TK, lo_all / TK);
  x.n_tiles = t_end - x.t_begin;
  if (x.n_tiles <= 0)                                    // no row sees a key of this chunk
    for (int n = lane; n < x.rows; n += 32)
      a.partials[((int64_t)x.u * a.n_chunks + x.chunk) * a.rows_max + x.row0 + n] = make_float2(-INFINITY, 0.f);
  return x;
}

// 64 rows of the item from row n0 on into half a block of a stage, as the TMA unit would lay them out (128-byte swizzle); zeros where
// the item has no row.  For what is no box of whole groups: the ragged end of a window, and groups that do not divide 64.  Asynchronous
// copies without registers: the whole half block is in flight at once.  Called by a whole warp.
// (Few instructions count: beside the epilogue the producer gets an issue slot every several cycles.)
template <int NH>
__device__ __forceinline__ void lse_q_rows(const ScoreArgs& a, const LseItem& x, uint32_t dst, int n0, int lane) {
  constexpr int RPI = 32 / (8 * NH);                          // rows per step of the warp
  const int G = a.group, live = min(x.rows - n0, 64);
  int off[2];                                                 // where the rows lane and lane + 32 begin, from the window's first token on
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int n = x.row0 + n0 + min(lane + 32 * i, live - 1), w = n / G;
    off[i] = (w * a.n_q_heads + (n - w * G)) * (64 * NH);
  }
  const int r = lane / (8 * NH), c = lane % (8 * NH);
  const __nv_bfloat16* src = a.q + (((int64_t)x.slab * a.sum_win + x.w0) * a.n_q_heads + x.layer_h * G) * (64 * NH) + c * 8;
  const uint32_t d = dst + (c >> 3) * HALF_BYTES + r * 128 + (((c & 7) ^ r) << 4);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
#pragma unroll 4
    for (int k = 0; k < 32; k += RPI) {
      const int o = __shfl_sync(0xffffffffu, off[i], k + r), row = 32 * i + k;
      cp_async16((d ^ ((k & 7) << 4)) + row * 128, src + o, row + r < live ? 16u : 0u);
    }
  }
}

// The shares (group, column half, and lane of a block held twice) of each row of a finished item; stores (reference in log2 units, sum),
// (-inf, 0) when the row saw no key of this chunk.  Called by a whole warp.
__device__ __forceinline__ void lse_merge(const float2 (&state)[2][LSE_MB][2][128], float2* dst, int rows, int lane) {
  const int n_half = (rows + 63) / 64;
  for (int n = lane; n < rows; n += 32) {
    const int i2 = n >> 6;                                    // half block
    const bool dup = (n_half & 1) && i2 == n_half - 1;
    float2 o[8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
      o[i] = i < 4 || dup ? state[i & 1][i2 >> 1][(i >> 1) & 1][(n & 127) + (i >> 2) * 64] : make_float2(-INFINITY, 0.f);
    float mm = -INFINITY;
#pragma unroll
    for (int i = 0; i < 8; ++i) mm = fmaxf(mm, o[i].x);
    float ss = 0.f;
    if (mm > -INFINITY) {
#pragma unroll
      for (int i = 0; i < 8; ++i) ss += o[i].x > -INFINITY ? o[i].y * exp2f(o[i].x - mm) : 0.f;
    }
    dst[n] = make_float2(mm, ss);
  }
}

// NH: 64-dim halves of the head dimension (head_dim = 64 NH); a K tile is NH x [128 keys][64 bf16].
// REGS: what the epilogue carries of all blocks of an item stays in registers (lse_moves).
template <int NPOLY, int NH, bool WIN, bool REGS>
__global__ void __launch_bounds__(LSE_THREADS, 1)
score_tc_lse_kernel(const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap qmap, const TcArgs ta,
                    const Exp2Cubic cubic) {
  pdl_begin();
  extern __shared__ __align__(1024) uint8_t smem[];
  constexpr int S = lse_stages(NH);
  constexpr int QCOLS = 32 * NH;                         // TMEM columns of a Q block
  static_assert(LSE_MB * QCOLS <= LSE_A_COLS, "Q columns");
  const ScoreArgs& a = ta.a;
  const int G = a.group;

  const uint32_t smem_base = smem_u32(smem);
  const uint32_t k_smem = smem_base;                               // S stages of a K tile
  LseBarriers* bars = reinterpret_cast<LseBarriers*>(smem + (size_t)S * (NH * HALF_BYTES));
  volatile int* abort_flag = &bars->abort_flag;
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // warp-uniform

  if ((smem_base & 1023u) != 0) {                                  // swizzled tiles need 1024-byte alignment
    if (threadIdx.x == 0) report(a.status, ACTKV_E_CUDA, -2, (int32_t)smem_base);
    return;
  }
  LseItem x_next;
  if (warp == 0) x_next = lse_item<WIN>(ta, blockIdx.x, lane);     // (its loads are under way while the others set up)
  if (threadIdx.x == 96) {
    for (int s = 0; s < S; ++s) { mbar_init(smem_u32(&bars->k_full[s]), 1); mbar_init(smem_u32(&bars->k_empty[s]), 2); bars->k_last[s] = RING_UNUSED; }
    for (int i = 0; i < LSE_ITEMS_AHEAD; ++i) {
      mbar_init(smem_u32(&bars->item_full[i]), 1);
      mbar_init(smem_u32(&bars->item_empty[i]), LSE_EPI_WARPS + 3);
    }
    for (int b = 0; b < LSE_SLOTS; ++b) {
      mbar_init(smem_u32(&bars->q_free[b]), 2);
      mbar_init(smem_u32(&bars->q_ready[b]), 1);
      mbar_init(smem_u32(&bars->tmem_full[b]), 1);
      mbar_init(smem_u32(&bars->tmem_empty[b]), LSE_EPI_WARPS / 2);
    }
    for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&bars->shares_full[i]), LSE_EPI_WARPS); mbar_init(smem_u32(&bars->shares_empty[i]), 1); }
    mbar_init(smem_u32(&bars->clc), 1);
    mbar_init(smem_u32(&bars->drained[0]), 1);
    mbar_init(smem_u32(&bars->drained[1]), 1);
    bars->abort_flag = 0;
    bars->at[0] = (int)blockIdx.x / ta.n_rg / a.n_chunks;
    bars->at[1] = (int)blockIdx.x / ta.n_rg % a.n_chunks;
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&bars->tmem_base), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = bars->tmem_base;

  // Every role walks the same items: the producer of warp 0 finds them and describes them in a small ring.  In the ring of stages an
  // item is its Q blocks, then its K tiles.
  if (warp == 0 || warp == 2) {
    // ---------------- TMA producers: alternate entries of the ring; warp 0 also finds the items ----------------
    const int p = warp >> 1;
    int e = 0, slot = 0;
    uint32_t ipar = 0, cpar = 0;
    bool ok = true;
    for (;;) {
      LseItem x;
      if (p == 0) {
        if (lane == 0) {
          mbar_expect_tx(smem_u32(&bars->clc), 16);
          clc_request(smem_u32(bars->clc_resp), smem_u32(&bars->clc));
        }
        __syncwarp();
        x = x_next;
        if (x.n_tiles > 0) {
          ok = mbar_wait_warp(smem_u32(&bars->item_empty[slot]), ipar ^ 1u, abort_flag, ta.wait_cycles);
          if (ok && lane == 0) {
            bars->item[slot] = x;
            mbar_arrive(smem_u32(&bars->item_full[slot]));
          }
        }
      } else {
        ok = mbar_wait_warp(smem_u32(&bars->item_full[slot]), ipar, abort_flag, ta.wait_cycles);
        if (!ok) break;
        x = bars->item[slot];
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars->item_empty[slot]));
        if (x.n_tiles <= 0) break;
      }
      if (ok && x.n_tiles > 0) {
        if (++slot == LSE_ITEMS_AHEAD) { slot = 0; ipar ^= 1u; }
        const int n_half = (x.rows + 63) / 64, n_mb = (n_half + 1) / 2;
        for (int b = 0; b < n_mb && ok; ++b, ++e) {
          if ((e & 1) != p) continue;
          const int s = ring_stage(e, S);
          ok = mbar_wait_warp(smem_u32(&bars->k_empty[s]), ring_parity(e, S) ^ 1u, abort_flag, ta.wait_cycles);
          if (!ok) break;
          // The two halves of the block; a last half that stands alone is held twice.  Whole groups all of whose rows the item has
          // come as TMA boxes.  Lanes without a row hold zeros: they take part in the votes of the epilogue, so what they hold must be the
          // same in every run, and no other request's.
          const uint32_t bar = smem_u32(&bars->k_full[s]), dst = k_smem + s * (NH * HALF_BYTES);
          auto first_row = [&](int j) { return min(2 * b + j, n_half - 1) * 64; };
          auto is_box = [&](int j) { return 64 % G == 0 && first_row(j) + 64 <= x.rows; };
          const int n_box = (is_box(0) ? 1 : 0) + (is_box(1) ? 1 : 0);
          if (n_box < 2) {
            for (int j = 0; j < 2; ++j)
              if (!is_box(j)) lse_q_rows<NH>(a, x, dst + j * (HALF_BYTES / 2), first_row(j), lane);
            cp_async_wait_all();
            fence_proxy_async();                 // (the copies are read by tcgen05.cp)
            __syncwarp();
          }
          if (lane == 0) { bars->k_last[s] = ring_parity(e, S); mbar_expect_tx(bar, (uint32_t)(n_box * NH) * (HALF_BYTES / 2)); }
          __syncwarp();
          if (lane < 2 * NH && is_box(lane & 1)) {
            const int hf = lane >> 1, j = lane & 1;
            const int tok = x.slab * a.sum_win + x.w0 + (x.row0 + first_row(j)) / G;
            tma_load_3d(dst + hf * HALF_BYTES + j * (HALF_BYTES / 2), &qmap, bar, hf * 64, x.layer_h * G, tok);
          }
        }
        if (ok) {
          const int layer = a.layer_begin + x.slab, first = (p - e) & 1;
          if (ta.k5) ok = k_tile_producer<true, NH>(&kmap, a, bars, k_smem, S, x.r, x.layer_h, layer, x.L, x.t_begin, x.n_tiles, lane, abort_flag, first, 2, ta.wait_cycles, ta.stall_tile, e);
          else ok = k_tile_producer<false, NH>(&kmap, a, bars, k_smem, S, x.r, x.layer_h, layer, x.L, x.t_begin, x.n_tiles, lane, abort_flag, first, 2, ta.wait_cycles, ta.stall_tile, e);
          e += x.n_tiles;
        }
      }
      if (p == 0) {
        // (also after giving up: the answer lands in this CTA's shared memory)
        bool answered = mbar_wait_warp(smem_u32(&bars->clc), cpar, nullptr, ta.wait_cycles);
        cpar ^= 1u;
        // injected fault: the answer does not arrive (there is no second one to wait for; the roles that wait for the item do so longer)
        if (ta.stall_tile == STALL_ANSWER) answered = mbar_wait_warp(smem_u32(&bars->clc), cpar, nullptr, ta.wait_cycles / 4);
        if (!answered) {                         // the CTA it names may have been cancelled: nobody would do its item
          if (lane == 0) *abort_flag = 1;
          ok = false;
          mbar_wait_warp(smem_u32(&bars->clc), cpar ^ 1u, nullptr, DRAIN_LIMIT_CYCLES);
        }
        const int id = answered ? clc_answer(smem_u32(bars->clc_resp)) : -1;
        fence_proxy_async();                     // (the answer has been read before the next one is written)
        __syncwarp();
        if (!ok || id < 0) break;
        x_next = lse_item<WIN>(ta, id, lane);
      }
      if (!ok) break;
    }
    if (p == 0 && ok) {
      ok = mbar_wait_warp(smem_u32(&bars->item_empty[slot]), ipar ^ 1u, abort_flag, ta.wait_cycles);
      if (ok && lane == 0) {
        bars->item[slot].n_tiles = 0;
        mbar_arrive(smem_u32(&bars->item_full[slot]));
      }
    }
    __syncwarp();
  } else if (warp == 1 || warp == 3) {
    // ---------------- MMA issuers: A = Q block in TMEM, B = K tile in shared memory ----------------
    // Two warps, one per accumulator: warp 1 issues the even jobs into accumulator 0, warp 3 the odd jobs into accumulator 1; warp 1
    // also brings the Q blocks into tensor memory.  The whole warp runs the loop (waits stay warp-uniform); one elected lane issues.
    // Both wait for every entry of the ring and release it (tcgen05.commit after the last job of the tile, or a plain arrive).
    const int mw = warp >> 1;
    const uint32_t idesc = idesc_bf16(128, 128);
    const uint64_t desc0 = smem_desc_sw128(k_smem);
    const uint32_t full_bar = smem_u32(&bars->tmem_full[mw]), empty_bar = smem_u32(&bars->tmem_empty[mw]);
    const uint32_t d = tmem_base + LSE_A_COLS + mw * 128;
    const bool leader = elect_one();
    bool ok = true;
    int s = 0, slot = 0, qh = 0;
    uint32_t kpar = 0, ipar = 0, epar = 1u, qpar = 3u, rpar = 0;    // qpar: a bit per half (a fresh barrier passes with 1)
    // Warp 3 also merges: the shares of an item after its own second job of the next one, when the epilogue is about to finish or has
    // finished the item.  (With the epilogue warps meeting at the end of an item to merge it, items of 32 tiles of two blocks cost
    // 9 % over longer ones.)
    int m_rows = 0, m_sp = 0;                      // the item to be merged: rows (0: none), which `state`
    uint32_t m_par = 0;
    float2* m_dst = nullptr;
    auto merge = [&]() {
      if (!mbar_wait_warp(smem_u32(&bars->shares_full[m_sp]), m_par, abort_flag, ta.wait_cycles)) return false;
      lse_merge(bars->state[m_sp], m_dst, m_rows, lane);
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bars->shares_empty[m_sp]));
      m_rows = 0;
      m_sp ^= 1;
      m_par ^= (uint32_t)(m_sp == 0);
      return true;
    };
    for (;;) {
      ok = mbar_wait_warp(smem_u32(&bars->item_full[slot]), ipar, abort_flag, ta.wait_cycles);
      if (!ok) break;
      const int n_tiles = uni(bars->item[slot].n_tiles), rows = uni(bars->item[slot].rows);
      float2* dst = a.partials + ((int64_t)bars->item[slot].u * a.n_chunks + bars->item[slot].chunk) * a.rows_max + bars->item[slot].row0;
      if (mw == 0 && lane < 2 && n_tiles > 0) bars->at[lane] = lane == 0 ? bars->item[slot].u : bars->item[slot].chunk;
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bars->item_empty[slot]));
      if (n_tiles <= 0) break;
      if (++slot == LSE_ITEMS_AHEAD) { slot = 0; ipar ^= 1u; }
      const int n_mb = (rows + 127) / 128;
      // the Q blocks go to the half of the Q columns that the previous item does not use; three at head_dim 128 take the first part of the
      // other half too, and wait until that item's products are done
      const uint32_t q_col = (uint32_t)qh * (LSE_A_COLS / 2);
      auto q_block = [&](int b) { return tmem_base + ((q_col + b * QCOLS) & (LSE_A_COLS - 1)); };
      const bool both = n_mb * QCOLS > LSE_A_COLS / 2;
      if (mw == 0) {
        ok = mbar_wait_warp(smem_u32(&bars->q_free[qh]), (qpar >> qh) & 1u, abort_flag, ta.wait_cycles);
        if (ok && both) ok = mbar_wait_warp(smem_u32(&bars->q_free[qh ^ 1]), (qpar >> (qh ^ 1)) & 1u, abort_flag, ta.wait_cycles);
        if (!ok) break;
        qpar ^= both ? 3u : 1u << qh;
      }
      for (int b = 0; b < n_mb; ++b) {
        ok = mbar_wait_warp(smem_u32(&bars->k_full[s]), kpar, abort_flag, ta.wait_cycles);
        if (!ok) break;
        tc_fence_after();
        if (leader) {
          if (mw == 0) {
            const uint64_t desc_s = desc0 + (uint64_t)((s * (NH * HALF_BYTES)) >> 4);
#pragma unroll
            for (int kk = 0; kk < 4 * NH; ++kk)
              tmem_cp_k16(q_block(b) + kk * 8, desc_s + (uint64_t)(((kk >> 2) * HALF_BYTES + (kk & 3) * 32) >> 4));
            umma_commit(smem_u32(&bars->k_empty[s]));
            if (b == n_mb - 1) umma_commit(smem_u32(&bars->q_ready[qh]));
          } else {
            mbar_arrive(smem_u32(&bars->k_empty[s]));
          }
        }
        if (++s == S) { s = 0; kpar ^= 1u; }
      }
      // (a barrier per half: warp 1 may be two items ahead, and comes back to a half only when warp 3 is done with it)
      if (ok && mw == 1) ok = mbar_wait_warp(smem_u32(&bars->q_ready[qh]), (rpar >> qh) & 1u, abort_flag, ta.wait_cycles);
      rpar ^= 1u << qh;
      // (every item begins with accumulator 0, so that its sums do not depend on what this CTA did before)
      int job = 0, n_issued = 0, flip = 0;
      for (int it = 0; ok && it < n_tiles; ++it) {
        ok = mbar_wait_warp(smem_u32(&bars->k_full[s]), kpar, abort_flag, ta.wait_cycles);
        if (!ok) break;
        tc_fence_after();
        const uint64_t desc_s = desc0 + (uint64_t)((s * (NH * HALF_BYTES)) >> 4);
        bool mine = false;
        for (int i = 0; i < n_mb; ++i, ++job) {
          if ((job & 1) != mw) continue;
          ok = mbar_wait_warp(empty_bar, epar, abort_flag, ta.wait_cycles);
          if (!ok) break;
          epar ^= 1u;
          tc_fence_after();
          if (leader) {
            const uint32_t at = q_block(i ^ flip);
#pragma unroll
            for (int kk = 0; kk < 4 * NH; ++kk)
              umma_bf16_ts(d, at + kk * 8, desc_s + (uint64_t)(((kk >> 2) * HALF_BYTES + (kk & 3) * 32) >> 4), idesc,
                           kk > 0 ? 1u : 0u);
            umma_commit(full_bar);
          }
          mine = true;
          ++n_issued;
        }
        if (!ok) break;
        if (leader) {
          if (mine) umma_commit(smem_u32(&bars->k_empty[s]));
          else mbar_arrive(smem_u32(&bars->k_empty[s]));
        }
        if (++s == S) { s = 0; kpar ^= 1u; }
        flip ^= lse_flip(rows);
        if (mw == 1 && m_rows > 0 && n_issued >= 2) {
          ok = merge();
          if (!ok) break;
        }
      }
      if (ok && mw == 1 && m_rows > 0) ok = merge();
      if (!ok) break;
      m_rows = rows;
      m_dst = dst;
      if (leader) {
        umma_commit(smem_u32(&bars->q_free[qh]));
        if (both) umma_commit(smem_u32(&bars->q_free[qh ^ 1]));
      }
      qh ^= 1;
    }
    if (ok && mw == 1 && m_rows > 0) ok = merge();
    // drain: every MMA issued above has completed before TMEM is freed
    __syncwarp();
    if (leader) umma_commit(smem_u32(&bars->drained[mw]));
    __syncwarp();
    // (a tear-down wait: it does not end early because another role gave up)
    mbar_wait_warp(smem_u32(&bars->drained[mw]), 0, nullptr, ok ? ta.wait_cycles : DRAIN_LIMIT_CYCLES);
    __syncwarp();
  } else {
    // ---------------- epilogue warps ----------------
    const int quarter = warp & 3;                  // TMEM lanes this warp may touch
    const int k = (warp - LSE_EPI_WARP0) >> 2;     // 0..3
    const int grp = k >> 1;                        // accumulator / job parity this warp serves
    const int half = k & 1;                        // its columns: [64 half, 64 half + 64)
    const int rib = quarter * 32 + lane;           // TMEM lane
    const int upper = quarter >> 1;                // lanes 64 and up: the second half of a block
    const float c = a.scale_log2;
    const uint32_t tq = tmem_base + ((uint32_t)(quarter * 32) << 16) + LSE_A_COLS + grp * 128 + half * 64;
    int slot = 0, sp = 0;                          // sp: which `state`
    uint32_t ipar = 0, fpar = 0, spar = 0;
    for (;;) {
      bool ok = mbar_wait_warp(smem_u32(&bars->item_full[slot]), ipar, abort_flag, ta.wait_cycles);
      if (!ok) break;
      const LseItem* x = &bars->item[slot];
      const int n_tiles = x->n_tiles, rows = x->rows;
      if (n_tiles <= 0) break;
      const int n_half = (rows + 63) / 64, n_mb = (n_half + 1) / 2;
      const bool twice = n_half & 1;               // the last block holds its rows twice: a lane folds half as many columns of them
      // this thread's row in row block b, and the last key it sees (lanes without a row of this item: every key; their sums are dropped)
      auto row_of = [&](int b) { return (2 * b + (twice && b == n_mb - 1 ? 0 : upper)) * 64 + (rib & 63); };
      auto last_of = [&](int n) { return (a.causal && n < rows) ? (x->L - x->W + (x->row0 + n) / G) : (x->L - 1); };
      if (!mbar_wait_warp(smem_u32(&bars->shares_empty[sp]), spar ^ 1u, abort_flag, ta.wait_cycles)) break;
      // the most restricted row's last key, and the largest first key (0 unless the layer has a sliding window)
      int jfast = x->L - 1, jlmax = 0;
      for (int b = 0; b < n_mb; ++b) {
        const int n = row_of(b), jm = last_of(n);
        jfast = min(jfast, jm);
        if (WIN && a.win_left > 0 && n < rows) jlmax = max(jlmax, jm - a.win_left + 1);
        bars->state[sp][grp][b][half][rib] = make_float2(-INFINITY, 0.f);
      }
      const bool moves = lse_flip(rows) != 0 || n_mb == 3;
      const int n_jobs = n_tiles * n_mb, b_short = twice ? n_mb - 1 : -1;
      float2* st0 = &bars->state[sp][grp][0][half][rib];
      int key0 = (x->t_begin + (n_mb == 1 ? grp : 0)) * TK + half * 64;
      // A group that stays with one row block keeps its (reference, sum) in registers and has little left to count per job.  Two blocks
      // that change places, and three: the next job is of the block before this one, cyclically, and of the same tile only from the first
      // of three to the last.  REGS: ms is the next job's (reference, sum), m1 and m2 those of the jobs after it.
      int b = n_mb == 1 ? 0 : grp;
      bool wide = b != b_short;
      int off = wide ? 0 : upper * 32;
      const int step = n_mb == 1 ? 2 * TK : TK;
      float2 ms = make_float2(-INFINITY, 0.f), m1 = ms, m2 = ms;
      for (int j = grp; j < n_jobs; j += 2) {
        ok = lse_job<NPOLY, WIN>(bars, abort_flag, tq + off, grp, fpar, wide, [&]() { return last_of(row_of(b)); }, ms,
                                 jfast - key0 - off + 1, jlmax - key0 - off, a.win_left, key0 + off, c, cubic, ta.wait_cycles);
        if (!ok) break;
        fpar ^= 1u;
        key0 += step;
        if (moves) {
          if constexpr (!REGS) st0[b * (2 * 128)] = ms;
          if (b == 0 && n_mb == 3) key0 -= TK;
          b = (b == 0 ? n_mb : b) - 1;
          wide = b != b_short;
          off = wide ? 0 : upper * 32;
          if constexpr (REGS) {
            const float2 t = ms;
            ms = m1;
            if (n_mb == 3) { m1 = m2; m2 = t; } else m1 = t;
          } else {
            ms = st0[b * (2 * 128)];
          }
        }
      }
      if (REGS ? moves || grp < n_jobs : !moves && grp < n_jobs) st0[b * (2 * 128)] = ms;
      if (REGS && moves) {
        b = (b == 0 ? n_mb : b) - 1;
        st0[b * (2 * 128)] = m1;
        if (n_mb == 3) st0[(b == 0 ? 2 : b - 1) * (2 * 128)] = m2;
      }
      if (!ok) break;
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(smem_u32(&bars->shares_full[sp]));
        mbar_arrive(smem_u32(&bars->item_empty[slot]));
      }
      if (++slot == LSE_ITEMS_AHEAD) { slot = 0; ipar ^= 1u; }
      sp ^= 1;
      spar ^= (uint32_t)(sp == 0);
    }
  }
  // ---------------- teardown ----------------
  tc_fence_before();
  __syncthreads();
  if (warp == 0 && lane == 0 && *abort_flag) {
    report(a.status, ACTKV_E_TIMEOUT, bars->at[0], bars->at[1]);
    drain_loads(bars, S);
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

}  // namespace tc
}  // namespace actkv
