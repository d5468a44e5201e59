// tickets.h -- which requests of the batch engine are queued, running or done,
// and the least buffers it runs them with.  Plain C++ (a test exercises it
// without a GPU).
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <unordered_map>
#include <vector>

namespace f12engine {

struct TicketState {
  bool done = false;
  int rc = 0;
  int batch = -1;                 // staging buffer of the batch that runs it
};

// No request queued or running.  A batch is launched in several passes, or
// captured first: until its last launch its tickets are not in `inflight`, and
// the event of its staging buffer is still the one of an earlier batch, so the
// event says something about the tickets in flight only.
template <class EventDone>
bool tickets_idle(const std::unordered_map<uint64_t, TicketState> &tickets, const std::vector<uint64_t> *inflight,
                  EventDone event_done) {
  for (const auto &kv : tickets) {
    const TicketState &t = kv.second;
    if (t.done) continue;
    if (t.batch < 0) return false;
    const std::vector<uint64_t> &f = inflight[t.batch];
    if (std::find(f.begin(), f.end(), kv.first) == f.end() || !event_done(t.batch)) return false;
  }
  return true;
}

// Doubles of Hermite rows with which any admitted request can run, outer pair
// by outer pair: a quartet of at most icap primitive quartets, whose inner side
// is the smaller one past 256 pairs, at the 680 doubles of order 14.
inline int64_t rows_least(int64_t icap) {
  const int64_t inner = std::max<int64_t>(256, (int64_t)std::ceil(std::sqrt((double)icap)));
  return 680 * std::min(icap, inner);
}

}  // namespace f12engine
