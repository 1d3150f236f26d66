// lclb_barrier.h -- the barrier of the blocks of one cooperative launch.
//
// Two words: the arrivals of the running barrier, zero between barriers, and a
// generation that each barrier advances by one.  Neither is ever compared for
// size, so a generation that wraps at 2^32 is no different from any other (an
// arrival counter that only grew met its wrap after 4.7 million
// re-discretisations of 152 blocks, which do not divide 2^32).  The wait is
// bounded: after spin_limit polls, or when another wait has already given up,
// the error word is set and the block gives up.
// M holds the two words and the error word (device atomics in k_rediscretise,
// std::atomic in the host test).
#pragma once

#ifdef __CUDACC__
#define LCLB_HD __host__ __device__ __forceinline__
#else
#define LCLB_HD inline
#endif

namespace lclb {

template <typename M>
LCLB_HD bool barrier_wait(M& m, unsigned nblocks, int spin_limit) {
  const unsigned gen = m.generation();  // before arriving: it cannot advance without this arrival
  if (m.arrive() == nblocks - 1) {
    m.clear_arrivals();
    m.advance();
    return true;
  }
  for (int spin = 0;; ++spin) {
    if (m.generation() != gen) return true;
    if (spin >= spin_limit || ((spin & 255) == 255 && m.failed())) break;
    m.pause();
  }
  m.fail();
  return false;
}

}  // namespace lclb
