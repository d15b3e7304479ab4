// The allocation-free residual's calls: where a call's outcome reaches the
// host, and how its last CTA is found.  Compiles without CUDA too, so that it
// can be tested on any machine.
#pragma once

#include <cstddef>
#include <cstdint>

#ifdef __CUDACC__
#define OPM_HOST_DEVICE __host__ __device__
#else
#define OPM_HOST_DEVICE
#endif

namespace opm {

constexpr int kNoallocDevices = 64;

// A device's words in the library's static memory, which the first call
// registers with CUDA.  Every device has a line of its own: host threads that
// serve one GPU each call at the same time.
// Both words hold a call's tag (with its result in outcome), so that no call
// takes another's.
struct alignas(128) NoallocLine {
  volatile uint64_t outcome;  // noalloc_outcome
  volatile uint32_t spoilt;   // a CTA's ticket was not one of this call's
};

// Registered as a whole, so it shares no page (up to 64 KB) with other data.
constexpr size_t kNoallocPage = 65536;
struct alignas(kNoallocPage) NoallocPage {
  NoallocLine line[kNoallocDevices];
};

constexpr uint32_t kNoallocDone = 1, kNoallocFault = 2;
OPM_HOST_DEVICE inline uint64_t noalloc_outcome(uint32_t tag, uint32_t result) { return (uint64_t)tag << 32 | result; }

// A device's ticket counter runs on from call to call: a call of t CTAs takes
// t tickets from base, the tickets of all earlier calls, and nothing is reset.
// So calls that overlap (which spoils their norms) leave the counter right
// for the next one.  Where the device's count is not what the host takes it
// to be (a launch that was recorded instead of run), a CTA sees a ticket
// outside the call's range, the call fails, and the next one starts with
// cleared words.
struct NoallocCall {
  uint32_t base, tag;
  bool clear;  // the device's words have to be cleared first
};

struct NoallocCalls {
  uint32_t tickets = 0, tag = 0;
  bool unsure = false;
  NoallocCall begin(uint32_t ctas) {
    const bool clear = unsure;
    if (clear) tickets = 0;
    unsure = false;
    if (++tag == 0) ++tag;  // 0: no call
    const NoallocCall c{tickets, tag, clear};
    tickets += ctas;
    return c;
  }
};

OPM_HOST_DEVICE inline bool noalloc_is_last(uint32_t ticket, uint32_t base, uint32_t ctas) {
  return ticket - base == ctas - 1;
}
OPM_HOST_DEVICE inline bool noalloc_is_foreign(uint32_t ticket, uint32_t base, uint32_t ctas) {
  return ticket - base >= ctas;
}

}  // namespace opm
