// Arithmetic of a ring of S stages in shared memory that two producers fill in turn: entry e is producer e % 2's, goes to stage e % S and
// completes that stage's (e / S)-th phase.  Plain C++ without CUDA headers, so that a host compiler takes it too.
#pragma once

#ifdef __CUDACC__
#define ACTKV_RING __host__ __device__ __forceinline__
#else
#define ACTKV_RING inline
#endif

namespace actkv {

ACTKV_RING int ring_stage(int e, int S) { return e % S; }
ACTKV_RING unsigned ring_parity(int e, int S) { return (unsigned)(e / S) & 1u; }     // to wait for on the stage's barrier
// Calls wait(stage, parity) for the last load that each stage was given, when producer p of two has issued its entries below end[p] and
// no others.  (The stage of entry e is filled again only after everyone has taken e out, so the two ends differ by S at most.)
template <class Wait>
ACTKV_RING void ring_drain(const int (&end)[2], int S, Wait wait) {
  const int hi = end[0] > end[1] ? end[0] : end[1];
  for (int e = hi > S ? hi - S : 0; e < hi; ++e) {
    const int last = e < end[e & 1] ? e : e - S;
    if (last >= 0) wait(ring_stage(last, S), ring_parity(last, S));
  }
}

}  // namespace actkv
