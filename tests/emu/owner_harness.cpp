// Test infrastructure: JoinOwners (join_owner.h) under threads that claim sets for
// the ids of a few streams.  Returns 0, or what went wrong.
#include <thread>
#include <vector>

#include "join_owner.h"

using namespace gbfft;

extern "C" int owners_run(int threads, int ids, int rounds) {
  for (int r = 0; r < rounds; ++r) {
    JoinOwners o;
    std::vector<std::vector<int>> got(threads, std::vector<int>(2 * ids));
    std::vector<std::thread> t;
    for (int k = 0; k < threads; ++k)
      t.emplace_back([&, k] {
        for (int j = 0; j < 2 * ids; ++j) got[k][j] = o.claim((uint64_t)((j + k + r) % ids));
      });
    for (auto& x : t) x.join();
    std::vector<int> set(ids, -2), of(kJoinSets, -1);
    for (int k = 0; k < threads; ++k)
      for (int j = 0; j < 2 * ids; ++j) {
        const int id = (j + k + r) % ids, s = got[k][j];
        if (s < -1 || s >= kJoinSets) return 1;
        if (set[id] == -2) set[id] = s;
        if (set[id] != s) return 2;                        // a stream's set never changes
        if (s >= 0 && of[s] >= 0 && of[s] != id) return 3;  // and is no other's
        if (s >= 0) of[s] = id;
      }
    for (int s = 0; s < kJoinSets; ++s)
      if ((of[s] >= 0) != (s < ids)) return 4;  // as many as there are ids are taken
  }
  return 0;
}
