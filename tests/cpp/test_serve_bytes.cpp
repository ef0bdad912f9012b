// Admission with and without the depth pass's byte per point (no GPU): the
// bytes never keep a request out that could have run.  Built and run by
// tests/test_serve_bytes.py.
#include <algorithm>
#include <cstdio>
#include <utility>
#include <vector>

#include "serve_core.h"

using adop::serve::RangeAllocator;
using adop::serve::bytes_cost_no_request;

// How many of `reqs` (state, points) are admitted in order, and how many got their bytes.
static std::pair<int, int> admit(const std::vector<std::pair<size_t, size_t>>& reqs, size_t pool, size_t run, int slots,
                                 bool with) {
  RangeAllocator a(pool, 256);
  size_t state = 0, bytes = 0;
  int active = 0, got = 0;
  for (const auto& r : reqs) {
    if (active >= slots || a.alloc(r.first) == SIZE_MAX) break;
    ++active;
    state += a.round(r.first);
    bytes += a.round(r.second);
    if (with &&
        bytes_cost_no_request(a.capacity(), a.in_use(), run, (size_t)slots, (size_t)active, state, bytes,
                              a.round(r.second)) &&
        a.alloc(r.second) != SIZE_MAX)
      ++got;
  }
  return {active, got};
}

int main() {
  const size_t M = 1000000;
  int granted = 0, refused = 0;
  for (size_t state : {1 * M, 18 * M, 121 * M, 486 * M})
    for (size_t n : {1 * M, 8 * M, 50 * M, 120 * M})
      for (size_t pool : {500 * M, 1200 * M, 6442 * M, 60000 * M})
        for (int slots : {1, 8, 64})
          for (size_t streams_batch : {1, 16, 32}) {
            const size_t run = std::min((size_t)slots, streams_batch);
            const std::vector<std::pair<size_t, size_t>> reqs(64, {state, n});
            const auto w = admit(reqs, pool, run, slots, true), o = admit(reqs, pool, run, slots, false);
            const int need = std::min((int)run, o.first);
            if (w.first < need) {
              std::printf("state %zu n %zu pool %zu slots %d run %zu: %d admitted, %d without the bytes\n", state, n,
                          pool, slots, run, w.first, o.first);
              return 1;
            }
            w.second == w.first ? ++granted : ++refused;  // all with their bytes, or some without
          }
  if (granted < 50 || refused < 50) return std::printf("granted %d, refused %d\n", granted, refused), 1;
  // small views of a large cloud: everything that fitted still does
  const auto small = admit(std::vector<std::pair<size_t, size_t>>(64, {18 * M, 120 * M}), 1200 * M, 32, 64, true);
  if (small.first != 64 || small.second != 0) return std::printf("small: %d, %d\n", small.first, small.second), 1;
  // a single large view of a large cloud takes them, in a pool that holds seventeen such views
  const auto one = admit({{486 * M, 50 * M}}, 8590 * M, 32, 64, true);
  if (one.first != 1 || one.second != 1) return std::printf("one: %d, %d\n", one.first, one.second), 1;
  // and up to seventeen of these views are admitted as before
  const std::vector<std::pair<size_t, size_t>> large(64, {486 * M, 50 * M});
  if (admit(large, 8590 * M, 32, 64, true).first != admit(large, 8590 * M, 32, 64, false).first) return 1;
  // a burst of mixed sizes over a cloud of 8M points has room for all bytes
  std::vector<std::pair<size_t, size_t>> mixed;
  for (int k = 0; k < 16; ++k) mixed.push_back({(size_t[]){18 * M, 54 * M, 121 * M, 486 * M}[k % 4], 8 * M});
  const auto m = admit(mixed, 6442 * M, 32, 64, true);
  if (m.first != 16 || m.second != 16) return std::printf("mixed: %d, %d\n", m.first, m.second), 1;
  std::printf("serve bytes: ok\n");
  return 0;
}
