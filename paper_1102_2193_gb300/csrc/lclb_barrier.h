// lclb_barrier.h -- the barrier of the blocks of one cooperative launch.
//
// One word: its top bit is the side of the barrier, the rest counts arrivals.
// All blocks but one add 1, that one adds what makes the sum of a barrier 2^31,
// so that the last arrival, whichever it is, flips the top bit and leaves the
// rest zero (sense reversal).  Nothing grows, so nothing wraps (an arrival counter
// that only grew met its wrap after 4.7 million re-discretisations of 152 blocks,
// which do not divide 2^32), and a block sends one atomic per barrier (a count and
// a generation apart, with the last block clearing one and advancing the other,
// took 10 us more of a step with seven barriers).  The wait is bounded: after
// spin_limit polls, or when another wait has already given up, the error word is
// set and the block gives up.
// M holds the word and the error word (device atomics in k_rediscretise,
// std::atomic in the host test).
#pragma once

#ifdef __CUDACC__
#define LCLB_HD __host__ __device__ __forceinline__
#else
#define LCLB_HD inline
#endif

namespace lclb {

template <typename M>
LCLB_HD bool barrier_wait(M& m, unsigned nblocks, bool first, int spin_limit) {
  const unsigned side = 0x80000000u, old = m.arrive(first ? side - (nblocks - 1) : 1u);
  for (int spin = 0;; ++spin) {
    if ((m.word() ^ old) & side) return true;
    if (spin >= spin_limit || ((spin & 255) == 255 && m.failed())) break;
    m.pause();
  }
  m.fail();
  return false;
}

}  // namespace lclb
