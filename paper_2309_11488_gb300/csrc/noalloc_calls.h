// Host side of the allocation-free residual's calls: where a call's outcome
// reaches the host.  Without CUDA, so that it can be tested on any machine.
#pragma once

#include <cstddef>

namespace opm {

constexpr int kNoallocDevices = 64;

// A device's words in the library's static memory, which the first call
// registers with CUDA.  Every device has a line of its own: host threads that
// serve one GPU each call at the same time.
struct alignas(128) NoallocLine {
  volatile unsigned int outcome;
};

// Registered as a whole, so it shares no page (up to 64 KB) with other data.
constexpr size_t kNoallocPage = 65536;
struct alignas(kNoallocPage) NoallocPage {
  NoallocLine line[kNoallocDevices];
};

}  // namespace opm
