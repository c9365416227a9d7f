// How the thread blocks that share a sequence settle its status word.
//
// The sequence has a 64-bit word in the workspace, zero between calls: below, how many of its blocks are through their
// roles; above, what went wrong until then (1: malformed input, put there by the block that looks; kFailed for every block in
// which a wait ran out).  A block adds itself once, and whoever completes the count publishes the status, from the one
// round trip of that addition, and clears the word.
//
// A wait that runs out later, in the merge, adds its mark to the word.  If blocks are still missing, the last of them finds
// it.  If none is, the mark came too late for the publisher: if that has cleared the word already, the block takes its mark off
// again, otherwise the mark goes with the rest, and the block waits for it (the publisher is past its roles, so it is
// running and waits for nothing but its last product).  Then it corrects what the publisher wrote.
// (The word is cleared by a store: with an addition that took off what the publisher had found, 4 x 64 nodes x 4096 keys took
// 23.88 us launch to launch instead of 23.71.)
// No order of these steps loses a failure or leaves the word other than zero, whatever the status word held before.
//
// `Words` is the memory: add(v) adds to the word and returns what it was, count() is its lower half, clear() makes it zero,
// put(s) writes the status, fence() orders what is before it ahead of what is behind it, correct() turns CLV_OK into CLV_ERR_TIMEOUT,
// expired() bounds the wait.
#pragma once

#include "clv.h"

#ifdef __CUDACC__
#define CLV_DEVICE __device__ __forceinline__
#else
#define CLV_DEVICE inline
#endif

namespace clv {

constexpr unsigned long long kFailed = 2ull << 32;

// a block is through its roles: what the word holds with it
template <class Words>
CLV_DEVICE unsigned long long add_block(Words& w, bool failed) {
  const unsigned long long mine = failed ? kFailed + 1ull : 1ull;
  return w.add(mine) + mine;
}
// by every block, with what add_block returned
template <class Words>
CLV_DEVICE void publish_if_last(Words& w, unsigned long long found, unsigned blocks) {
  if ((unsigned)found != blocks) return;
  const unsigned wrong = (unsigned)(found >> 32);
  w.put((wrong & 1u) ? CLV_ERR_TREE : wrong ? CLV_ERR_TIMEOUT : CLV_OK);
  w.fence();
  w.clear();
}
// a wait behind add_block ran out (and behind publish_if_last, if this block is the last)
template <class Words>
CLV_DEVICE void report_late(Words& w, unsigned blocks) {
  const unsigned there = (unsigned)w.add(kFailed);
  if (there != 0u && there != blocks) return;
  if (there == 0u) w.add(0ull - kFailed);
  while (w.count() != 0u && !w.expired()) {}
  w.fence();
  w.correct();
}

}  // namespace clv
