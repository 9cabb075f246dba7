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
// A parity that a fresh barrier passes: nothing was ever loaded into the stage.  The producers record each load's parity, so that the
// tear-down waits for what may still be in flight.
constexpr unsigned RING_UNUSED = 1u;

}  // namespace actkv
