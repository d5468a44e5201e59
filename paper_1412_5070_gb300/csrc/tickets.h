// tickets.h -- which requests of the batch engine are queued, running or done.
// Plain C++ (a test exercises it without a GPU).
#pragma once

#include <algorithm>
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

}  // namespace f12engine
