// The ring of slots through which a block of the star solve reads its records: record i lies in
// slot i % SLOTS, and its arrival completes phase i / SLOTS of the slot's mbarrier.  Host and
// device code without CUDA headers, so that the order can be checked by a host program.
#pragma once

#ifdef __CUDACC__
#define RING_FN __host__ __device__ inline
#else
#define RING_FN inline
#endif

namespace spnet {

constexpr int SLOTS = 3;

// Records asked for by the time the block waits for record `rec`: the first SLOTS at the start,
// record rec - 1 + SLOTS once the wait for rec > 0 is over (its slot is free then).
RING_FN int ring_issued(int rec, int nrec) {
  const int n = rec > 0 ? rec - 1 + SLOTS : SLOTS;
  return n < nrec ? n : nrec;
}
RING_FN unsigned ring_parity(int rec) { return (unsigned)(rec / SLOTS) & 1u; }

}  // namespace spnet
