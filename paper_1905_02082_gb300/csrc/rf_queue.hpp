// Queue of a batch's registrations: how the groups of CTAs of one cooperative
// launch take the batch's streams (host and device code, no CUDA calls: the
// memory operations come with `Mem`, so the protocol also runs on host
// threads).
//
// Group g starts with queue position g.  When it has registered position `at`,
// its leader takes the next position from the shared counter and publishes it
// in links[at]; the other members follow that link.  A link is written once,
// by a compare-and-swap from kLinkNone: either the leader's position + 1, or
// kLinkClosed by a member that has waited too long, whichever comes first.
// All members therefore read the same link, also those that arrive late, and
// every position is registered by all members of one group or by none: the
// counts by which a registration ends stay complete.  (One word per group,
// overwritten for every stream, let a member give up while the leader went
// on: the streams that followed never saw their last member leave.)
//
// Positions that no group registers are given to Mem::abandon, once each: the
// one that the leader had taken when it found its link closed, and, when no
// group is left, the rest of the queue.
#pragma once

#ifndef RF_HD
#ifdef __CUDACC__
#define RF_HD __host__ __device__ __forceinline__
#else
#define RF_HD inline
#endif
#endif

namespace rf {

constexpr unsigned kLinkNone = 0u, kLinkClosed = ~0u;

// The leader's next position after `at`; n when the group ends.
template <class Mem>
RF_HD int queue_lead(Mem& m, unsigned* links, unsigned* counter, unsigned* groups_left, int at, int n) {
  const int taken = (int)m.add(counter, 1u);
  const int next = taken < n ? taken : n;
  if (m.cas(links + at, kLinkNone, (unsigned)next + 1u) == kLinkNone) return next;
  if (next < n) m.abandon(next);
  if (m.add(groups_left, ~0u) == 1u)  // (- 1: the last group that could take them)
    for (int k; (k = (int)m.add(counter, 1u)) < n;) m.abandon(k);
  return n;
}

// Another member's next position after `at`; n when the group ends.  At most
// `limit` polls.
template <class Mem>
RF_HD int queue_follow(Mem& m, unsigned* links, int at, int n, long long limit) {
  unsigned w;
  for (long long spins = 0; (w = m.load(links + at)) == kLinkNone;) {
    if (++spins > limit) {
      w = m.cas(links + at, kLinkNone, kLinkClosed);
      if (w == kLinkNone) w = kLinkClosed;
      break;
    }
    m.pause(spins);
  }
  return w == kLinkClosed ? n : (int)w - 1;
}

}  // namespace rf
