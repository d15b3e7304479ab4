// The bookkeeping of the allocation-free residual's calls, with no GPU.
#include <cstdint>
#include <cstdio>
#include <vector>

#include "noalloc_calls.h"

using namespace opm;

#define EXPECT(c) \
  if (!(c)) return printf("line %d: %s\n", __LINE__, #c), 1

static NoallocPage page;

// Two GPUs' calls at once: neither clears nor reads the other's outcome.
static int outcomes_per_device() {
  for (int a = 0; a < kNoallocDevices; ++a) {
    for (int b = 0; b < kNoallocDevices; ++b) page.line[b].outcome = 1u + b;
    page.line[a].outcome = 0u;
    for (int b = 0; b < kNoallocDevices; ++b) EXPECT(page.line[b].outcome == (a == b ? 0u : 1u + b));
  }
  EXPECT((uintptr_t)&page % kNoallocPage == 0 && sizeof(page) % kNoallocPage == 0);
  return 0;
}

// One CTA's arrival, as the kernel does it.
struct Gpu {
  uint32_t counter = 0;
  int last = 0, foreign = 0;
  void arrive(const NoallocCall &c, uint32_t ctas) {
    const uint32_t t = counter++;
    last += noalloc_is_last(t, c.base, ctas);
    foreign += noalloc_is_foreign(t, c.base, ctas);
  }
  // A call on its own: it succeeds if its last arrival, and no other, is the last CTA.
  bool run(NoallocCalls &h, uint32_t ctas) {
    const NoallocCall c = h.begin(ctas);
    if (c.clear) counter = 0;
    last = foreign = 0;
    bool early = false;
    for (uint32_t q = 0; q < ctas; ++q) {
      early = early || last > 0;
      arrive(c, ctas);
    }
    if (foreign || last != 1) h.unsure = true;
    return !early && last == 1 && foreign == 0;
  }
};

// After two calls that overlapped in any order of arrivals, the next call is right.
static int next_call_after_overlap() {
  for (uint32_t m = 1; m <= 4; ++m)
    for (uint32_t order = 0; order < 1u << 8; ++order) {
      Gpu g;
      NoallocCalls h;
      h.tickets = g.counter = 0xfffffffau;  // and across the counter's wrap
      const NoallocCall a = h.begin(4), b = h.begin(m);
      uint32_t na = 0, nb = 0;
      for (int q = 0; na + nb < 4 + m; ++q) {
        const bool take_a = nb == m || (na < 4 && (order >> q & 1u));
        g.arrive(take_a ? a : b, take_a ? 4 : m);
        ++(take_a ? na : nb);
      }
      EXPECT(g.run(h, 3) && g.run(h, 1) && g.run(h, 8));
    }
  return 0;
}

// A launch that was recorded and never ran: the call failed, the next one starts afresh.
static int launch_that_never_ran() {
  Gpu g;
  NoallocCalls h;
  EXPECT(g.run(h, 5));
  h.begin(7);
  h.unsure = true;
  EXPECT(g.run(h, 4) && g.run(h, 9));
  // unknown to the host: a call reports it instead of electing a wrong CTA, and the one after is right
  for (uint32_t lost : {1u, 3u, 100u}) {
    h.begin(lost);
    EXPECT(!g.run(h, 4) && g.run(h, 4));
    g.counter += lost;
    EXPECT(!g.run(h, 4) && g.run(h, 4));
  }
  return 0;
}

static int tags_differ() {
  NoallocCalls h;
  h.tag = 0xfffffffeu;
  const uint32_t a = h.begin(1).tag, b = h.begin(1).tag;
  EXPECT(a == 0xffffffffu && b == 1);  // 0 is no call's
  EXPECT(noalloc_outcome(a, kNoallocDone) >> 32 == a && (uint32_t)noalloc_outcome(a, kNoallocFault) == kNoallocFault);
  return 0;
}

int main() {
  return outcomes_per_device() || next_call_after_overlap() || launch_that_never_ran() || tags_differ();
}
