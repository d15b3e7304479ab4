// The host side of the allocation-free residual's calls, with no GPU.
#include <cstdint>
#include <cstdio>

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

int main() { return outcomes_per_device(); }
