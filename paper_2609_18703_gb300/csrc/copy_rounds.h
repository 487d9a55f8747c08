// copy_rounds.h — the rounds in which a copy CTA's producer warps take chunks
// (asm_copy).  Plain C++, so that the protocol can also be run on the host.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define RO_HD __host__ __device__ __forceinline__
#else
#define RO_HD inline
#endif

namespace ro {

// Lies in shared memory.  The producers meet at a barrier once a round.  Before
// round r's barrier producer 0 publishes the first chunk of round r + 1 (round
// 0's is set up front) and whether a wait of the CTA has given up; after it
// each producer asks leave(r), which reads published values only, so that all
// of them leave at the same round whatever happened to each one's own waits: a
// producer alone at the barrier would wait for good.  Producer 0 may be in
// front of round r + 1's barrier while another one still reads round r's
// values: rounds r to r + 2 have places of their own, and so have the flags of
// r and r + 1.
struct CopyRounds {
  uint32_t base[4];
  uint32_t stop[2];

  RO_HD void start(uint32_t first_chunk) { base[0] = first_chunk; }
  RO_HD void publish(uint32_t r, uint32_t next, uint32_t gave_up) {
    base[(r + 1u) & 3u] = next;
    stop[r & 1u] = gave_up;
  }
  RO_HD uint32_t chunk(uint32_t r) const { return base[r & 3u]; }   // of rounds r and r + 1, after r's barrier
  RO_HD bool leave(uint32_t r, uint32_t n_chunks) const {
    return base[r & 3u] >= n_chunks || stop[r & 1u] != 0u;
  }
};

}  // namespace ro
