// The device's look at the words the host writes, in an order that keeps what the host was promised.  Plain C++, so that
// the order can be checked on the CPU against every interleaving with the host's stores.
#pragma once
#include <stdint.h>

#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace blink {

struct MailboxView {
  uint32_t stop;
  bool started;
  uint64_t tail;   // submit entries published; what it says counts only when started
};

// `gated`: admission waits for the start word.  The host publishes a submit entry (sub_tail, release) before it sets
// start, and everything submitted before the start has to be visible to the first step: start is read before sub_tail,
// with acquire.  A loop that is not gated (never paused, or past its first step) reads stop and sub_tail in one round
// trip to host memory.
template <typename Words>
__host__ __device__ __forceinline__ MailboxView read_mailbox(Words& w, bool gated) {
  MailboxView v;
  v.stop = w.stop_relaxed();
  v.started = !gated || w.start_acquire() != 0u;
  v.tail = w.sub_tail_acquire();
  return v;
}

}  // namespace blink
