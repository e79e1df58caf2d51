// Bounded waits of the warp-specialised kernels, apart from what is polled (an mbarrier phase) and
// from what passes the time between polls, so that they run on the host as well.
#pragma once

#ifdef __CUDACC__
#define HELM6_HD __host__ __device__ __forceinline__
#else
#define HELM6_HD inline
#endif

namespace helm6 {

// A role's wait for another role: done() polls once, rest() passes the time until the next poll.
// False when another role has raised *fail (looked at every `look` polls, a power of two) or after
// `polls` polls, which raises it.
template <class Done, class Rest>
HELM6_HD bool wait_role(Done done, Rest rest, volatile int* fail, int polls, int look) {
  for (int it = 0; it < polls; ++it) {
    if (done()) return true;
    if ((it & (look - 1)) == look - 1 && *fail) return false;
    rest();
  }
  *fail = 1;
  return false;
}

// The wait for what the CTA itself has under way in the hardware (products, bulk copies) before it
// gives up the memory they use.  That completes whatever the other roles do, and it matters most
// after one of them has failed: *fail does not end this wait, completion or `polls` polls do.
template <class Done, class Rest>
HELM6_HD bool wait_flight(Done done, Rest rest, volatile int* fail, long long polls) {
  for (long long it = 0; it < polls; ++it) {
    if (done()) return true;
    rest();
  }
  *fail = 1;
  return false;
}

}  // namespace helm6
