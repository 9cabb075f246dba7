// Interval arithmetic of a lower-bound search by one warp, 32 probes at a time.  Plain C++ without CUDA headers, so that
// a host compiler takes it too.
//
// The answer (the first index whose entry is not below the key) lies in [lo, hi].  While hi - lo > 32, probe i of 0 .. 31 looks
// at search_probe(i); the list being ascending, the probes that find an entry below the key are a prefix of `below` probes.
#pragma once

#ifdef __CUDACC__
#define ACTKV_HD __host__ __device__ __forceinline__
#else
#define ACTKV_HD inline
#endif

namespace actkv {

struct SearchSpan {
  int lo, hi;
};
ACTKV_HD int search_step(SearchSpan s) { return (s.hi - s.lo + 32) / 33; }
ACTKV_HD int search_probe(SearchSpan s, int i) { return s.lo + (i + 1) * search_step(s) - 1; }      // (may be >= hi: not below)
// Only a probe that was not below bounds the answer from above: after 32 that were, it may still be hi.
ACTKV_HD SearchSpan search_narrow(SearchSpan s, int below) {
  SearchSpan t{s.lo + below * search_step(s), s.hi};
  if (below < 32 && search_probe(s, below) < s.hi) t.hi = search_probe(s, below);
  return t;
}

}  // namespace actkv
