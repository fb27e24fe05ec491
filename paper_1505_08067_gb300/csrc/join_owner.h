// Whose are a joined frame plan's counter sets: pure host logic, so that it can be
// tested without CUDA.
#pragma once
#include <stdint.h>

#include <atomic>

namespace gbfft {

// Frame plans have no workspace, so executions on several streams may overlap, and
// each stream needs counters of its own: a set belongs to the first stream that
// asks for it, for good (stream ids, unlike handles, are not used again).  Four
// sets: what a user's program has, a warm-up or a capture apart, and one for
// fft_execute_host's own stream.  Thread-safe.
constexpr int kJoinSets = 4;
class JoinOwners {
 public:
  // The set of stream `id`; -1 when all belong to others.
  int claim(uint64_t id) {
    for (int i = 0; i < kJoinSets; ++i) {
      uint64_t owner = 0;  // sets are taken in order, so no later one can be id's already
      if (of_[i].compare_exchange_strong(owner, id + 1) || owner == id + 1) return i;
    }
    return -1;
  }

 private:
  std::atomic<uint64_t> of_[kJoinSets] = {};  // id + 1; 0: free
};

}  // namespace gbfft
