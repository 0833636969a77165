// Arrivals at a registration's evaluations and the exit from it (host and
// device code, no CUDA calls: the memory operations come with `Mem`, so the
// protocol also runs in a host model of weakly ordered memory).
//
// One thread per CTA makes both calls.  An arrival is a relaxed reduction:
// the readers check the tags of what they read, so nothing waits for it.  The
// exit releases it: the last CTA of a large group need not itself have seen
// every arrival (register_body leaves out the last eighth of the count), and
// it stores 0 over the count, so every arrival has to come before its CTA's
// exit, and the last exit after all the others.  One access per registration.
#pragma once

#ifndef RF_HD
#ifdef __CUDACC__
#define RF_HD __host__ __device__ __forceinline__
#else
#define RF_HD inline
#endif
#endif

namespace rf {

template <class Mem>
RF_HD void arrive(Mem& m, unsigned* arrivals) {
  m.red_relaxed(arrivals, 1u);
}

// True on the last of G CTAs to leave.
template <class Mem>
RF_HD bool last_to_leave(Mem& m, unsigned* left, unsigned G) {
  return m.add_acq_rel(left, 1u) == G - 1u;
}

}  // namespace rf
