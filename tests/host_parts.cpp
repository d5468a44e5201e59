// host_parts.cpp -- CPU build of the library's host-side parts that need no
// CUDA, for tests.  The library never loads this file's build.
#include <cstdint>
#include <unordered_map>
#include <vector>

#include "../paper_1412_5070_gb300/csrc/hoststage.h"
#include "../paper_1412_5070_gb300/csrc/perdevice.h"
#include "../paper_1412_5070_gb300/csrc/scratchcut.h"
#include "../paper_1412_5070_gb300/csrc/screen.h"
#include "../paper_1412_5070_gb300/csrc/tickets.h"

extern "C" {

// One ticket: done or not, its staging buffer (-1: none yet), whether it is in
// flight there, and what the buffer's event says.
int host_tickets_idle(int done, int batch, int in_flight, int event_done) {
  std::unordered_map<uint64_t, f12engine::TicketState> t;
  t[7].done = done != 0;
  t[7].batch = batch;
  std::vector<uint64_t> f[2];
  if (in_flight) f[batch].push_back(7);
  return f12engine::tickets_idle(t, f, [&](int) { return event_done != 0; }) ? 1 : 0;
}

int64_t host_rows_least(int64_t icap) { return f12engine::rows_least(icap); }

// Values of a sequence of devices (fill counts its calls and fails the first
// time for device `bad`); returns the number of fills.
int host_per_device(const int *device, int n, int bad, int *value, int *status) {
  f12host::PerDevice<int> t;
  int fills = 0;
  bool failed = false;
  for (int i = 0; i < n; ++i)
    status[i] = t.get(device[i], &value[i], [&](int &v) {
      ++fills;
      if (device[i] == bad && !failed) {
        failed = true;
        return -6;
      }
      v = 100 + device[i];
      return 0;
    });
  return fills;
}

struct CountingPin {
  static inline int locks = 0, frees = 0;
  static bool alloc(void **p, size_t n) {
    ++locks;
    *p = std::malloc(n);
    return true;
  }
  static void free(void *p) {
    ++frees;
    std::free(p);
  }
};

// Grows a stage through n sizes, keeping its first byte; locks[0], [1]: pages
// locked and freed.  Returns 1 if the byte survived.
int host_stage(int may_pin, const int64_t *bytes, int n, int *locks) {
  CountingPin::locks = CountingPin::frees = 0;
  f12host::HostStage<CountingPin> s(may_pin != 0);
  int ok = 1;
  for (int i = 0; i < n; ++i) {
    if (!s.reserve((size_t)bytes[i], i ? 1 : 0)) return 0;
    if (i == 0) s.p[0] = 77;
    ok = ok && s.p[0] == 77;
  }
  s.release();
  locks[0] = CountingPin::locks;
  locks[1] = CountingPin::frees;
  return ok;
}

int host_scratch_cut(int64_t room, int direct, int64_t nf, int64_t big_pq, int64_t big_in, int64_t pitch,
                     int64_t *c) {
  f12host::ScratchCut s;
  const bool ok = f12host::scratch_cut(room, direct != 0, nf, 16, big_pq, big_in, pitch, &s);
  c[0] = s.keys_cap;
  c[1] = s.part_thin;
  c[2] = s.part_cap;
  c[3] = s.rows_cap;
  return ok ? 1 : 0;
}

int host_grow_index(float x, int n) { return f12k::grow_index(x, n); }

// n candidates against a table: 1 negligible, 0 not, as the kernels decide
// (got) and weighed in double precision (want); returns how many took both.
int host_screen(const double *g, int ng, double limit, const double *v, const double *u, const double *iv, int n,
                int *got, int *want) {
  std::vector<float> g32;
  for (int i = 0; i < ng; ++i) g32.push_back(g[i] < 3e38 ? (float)g[i] : INFINITY);
  const float band = f12k::screen_band(g, ng), lim = (float)std::log2(limit);
  int both = 0;
  for (int i = 0; i < n; ++i) {
    want[i] = f12k::screen_negligible(v[i], u[i], iv[i], limit, g, ng) ? 1 : 0;
    const int s = f12k::screen_single(v[i], u[i], iv[i], lim, g32.data(), ng, band);
    got[i] = s >= 0 ? s : want[i];
    both += s < 0;
  }
  return both;
}

}  // extern "C"
