// Allocation-free residual entry point.
//
// Some callers cannot allocate device memory at the point where they need a
// residual: code running inside a simulator's own memory pool or arena (which
// forbids foreign cudaMalloc calls), code called while the caller holds a
// fixed device-memory budget it must not exceed, or code in a process where
// every allocation goes through an allocator the library cannot see.  For
// them, opm_bsr_residual_noalloc computes r = b - A x and the 2-norms
// ||r||_2, ||b||_2 on the caller's own BSR arrays without creating a handle
// and without allocating anything.
//
// Its only scratch (one partial sum pair per CTA, the CTAs' ticket counter and
// a pattern-error word) is the file-scope array below: every GPU that loads
// the library holds these 131,328 bytes until the process exits, every call
// shares them, and they keep the last call's partial sums.  The counter runs
// on from call to call and the error word holds the tag of the call that set
// it, so no call depends on how an earlier one ended (noalloc_calls.h).
// The outcome reaches the host through the device's word in the library's own
// static memory, which the first call registers with CUDA (cudaHostRegister):
// a copy back into pageable memory took longer than a small residual.  Calls
// that overlap on one GPU (on two streams, or from two host threads) race on
// the array and give wrong results: serialise them.  Calls on different GPUs
// share nothing.
//
// The caller's pattern is not validated on the host (that would need a copy
// of it).  The kernel checks what it can before each access: a row whose
// start is negative or whose end lies before its start is taken as empty, a
// column outside [0, nb) is skipped; either sets the error word, the norms
// become NaN and the call returns OPM_ERR_PATTERN.  rowptr[nb] beyond the
// length of colidx and vals cannot be detected without that length: a
// well-formed pattern is the caller's precondition.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "../../include/opm_bsr.h"
#include "noalloc_calls.h"

namespace {

using opm::kNoallocDevices;
using opm::NoallocCall;
using opm::NoallocLine;

constexpr int kNaMaxRows = 2097152;
constexpr int kNaMaxTiles = 8192;              // CTAs of a call
constexpr int kNaThreads = 128;
constexpr int kNaWarps = kNaThreads / 32;
constexpr int kNaGroup = 10;                   // rows of a warp at a time, three lanes each
constexpr int kNaTile = kNaGroup * kNaWarps;   // rows of a CTA at a time
constexpr int kNaChunk = 72;                   // blocks of a group staged at a time
constexpr size_t kNaCounterBytes = 256;        // counter and error word, padded to their own lines
constexpr size_t kNaScratchBytes = kNaCounterBytes + sizeof(double) * 2 * kNaMaxTiles;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaScratchBytes];

std::mutex g_setup_mutex;
unsigned char *g_scratch_ptr[kNoallocDevices] = {};
opm::NoallocCalls g_calls[kNoallocDevices];

// Device address of the scratch array for the current device dev (looked up once
// per device, with that device current, and kept: calls after a
// cudaDeviceReset of that device are not supported, since the reloaded
// module may place the array elsewhere).
opm_status scratch_address(int dev, unsigned char **out) {
  if (dev < 0 || dev >= kNoallocDevices) return OPM_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  if (!g_scratch_ptr[dev]) {
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
      cudaGetLastError();
      return OPM_ERR_CUDA;
    }
    g_scratch_ptr[dev] = static_cast<unsigned char *>(p);
  }
  *out = g_scratch_ptr[dev];
  return OPM_OK;
}

// True for device (or managed) memory of device dev; host memory and another
// GPU's memory are refused.
bool on_device(const void *p, int dev) {
  cudaPointerAttributes at;
  if (!p || cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return (at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged) && at.device == dev;
}

// Copies eight bytes to shared memory in the background (cp.async.wait_all).
__device__ __forceinline__ void copy8_async(double *dst, const double *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// r = b - A x on the caller's BSR matrix (row-major 3x3 blocks); per-CTA
// partials of ||r||^2 and ||b||^2 in the scratch array, summed by the last
// CTA.  Pattern faults that can be seen from the row (see the file header)
// skip the access and set the error word to the call's tag; the last CTA then
// writes NaN norms.
//
// A warp takes groups of kNaGroup rows, three lanes per row, one component
// each (30 of 32 lanes at work on the FP64 pipe, which bounds the product:
// nine FMAs per 76 bytes).  The blocks of consecutive rows are contiguous, so
// the group's blocks, and the vector blocks that their columns name, are
// staged in shared memory with one wait for memory each.  Before, a thread
// per row read its blocks in place (a sector per lane and load, a wait for
// the columns and one for the vector at every block) and one thread summed
// all partials.  A group whose rows are not consecutive (a pattern fault)
// still reads its blocks in place.
// Measured, whole call: 2,590 rows 37.6 -> 26.8 us, 249,053 rows 173.9 -> 77.3,
// 949,871 rows 588.9 -> 196.3 (one group per warp: 115 and 272 for the last
// two, the sums' additions costing as much as the product).
__global__ void __launch_bounds__(kNaThreads, 8) k_residual_noalloc(
    int32_t nb, const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
    const double *__restrict__ vals, const double *__restrict__ x, const double *__restrict__ b,
    double *__restrict__ r, double *__restrict__ norms, unsigned char *scratch, NoallocLine *line, uint32_t base,
    uint32_t tag) {
  __shared__ double sv[kNaWarps][9 * kNaChunk];
  __shared__ double sx[kNaWarps][3 * kNaChunk];
  __shared__ double sm[2][kNaWarps];
  __shared__ unsigned int skip[kNaWarps][(kNaChunk + 31) / 32];  // blocks whose column is outside
  __shared__ int amlast;
  unsigned int *counter = reinterpret_cast<unsigned int *>(scratch);
  unsigned int *bad = counter + 1;
  double *partials = reinterpret_cast<double *>(scratch + kNaCounterBytes);
  const unsigned all = 0xffffffffu;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int row = lane / 3, comp = lane - 3 * row;  // lanes 30 and 31 have no row
  double rr = 0.0, bb = 0.0;
  bool fault = false;
  for (int64_t g = blockIdx.x;; g += gridDim.x) {
    const int64_t r0 = g * kNaTile + wp * kNaGroup;
    const int64_t i = r0 + row;
    const bool in = row < kNaGroup && i < nb;
    if (r0 >= nb) break;  // warp-uniform
    int m0 = in ? rowptr[i] : 0, m1 = in ? rowptr[i + 1] : 0;
    const double bi = in ? b[3 * i + comp] : 0.0;
    if (in && (m0 < 0 || m1 < m0)) {
      fault = true;
      m1 = m0;
    }
    // rows of a well-formed pattern follow one another
    const int next = __shfl_down_sync(all, m0, 3);
    const bool last = row == kNaGroup - 1 || i == nb - 1;
    const bool staged = !__any_sync(all, in && (fault || (!last && next != m1)));
    double y = 0.0;
    if (staged) {
      const int first = __shfl_sync(all, m0, 0);
      const int end = __reduce_max_sync(all, in ? m1 : first);
      for (int64_t c = first; c < end; c += kNaChunk) {  // past the last block, c may not fit an int32
        const int c0 = (int)c, cnt = min(kNaChunk, end - c0);
        constexpr int kV = (9 * kNaChunk + 31) / 32, kX = (3 * kNaChunk + 31) / 32, kS = (kNaChunk + 31) / 32;
        int col[kX];
#pragma unroll
        for (int q = 0; q < kX; ++q) {
          const int e = lane + 32 * q;
          col[q] = e < 3 * cnt ? colidx[c0 + e / 3] : 0;
        }
        __syncwarp();  // the last chunk has been read
#pragma unroll
        for (int q = 0; q < kV; ++q) {
          const int e = lane + 32 * q;
          if (e < 9 * cnt) copy8_async(&sv[wp][e], vals + 9ll * c0 + e);
        }
        if (lane < kS) skip[wp][lane] = 0;
        __syncwarp();
#pragma unroll
        for (int q = 0; q < kX; ++q) {
          const int e = lane + 32 * q;
          const bool out = col[q] < 0 || col[q] >= nb;
          if (out) {
            fault = true;
            atomicOr(&skip[wp][(e / 3) >> 5], 1u << ((e / 3) & 31));
          }
          if (e < 3 * cnt) sx[wp][e] = out ? 0.0 : x[3ll * col[q] + e % 3];
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        const int k1 = min(m1, c0 + cnt) - c0;
        for (int m = max(m0, c0) - c0; m < k1; ++m) {
          if ((skip[wp][m >> 5] >> (m & 31)) & 1u) continue;
          const double *a = sv[wp] + 9 * m + 3 * comp;
          const double *xj = sx[wp] + 3 * m;
          y = fma(a[0], xj[0], fma(a[1], xj[1], fma(a[2], xj[2], y)));
        }
      }
    } else {
      for (int m = m0; m < m1; ++m) {
        const int c = colidx[m];
        if (c < 0 || c >= nb) {
          fault = true;
          continue;
        }
        const double *a = vals + 9ll * m + 3 * comp;
        const double *xj = x + 3ll * c;
        y = fma(a[0], xj[0], fma(a[1], xj[1], fma(a[2], xj[2], y)));
      }
    }
    if (in) {
      const double d = bi - y;
      r[3 * i + comp] = d;
      rr = fma(d, d, rr);
      bb = fma(bi, bi, bb);
    }
  }
  if (fault) atomicExch(bad, tag);
  for (int o = 16; o > 0; o >>= 1) {
    rr += __shfl_xor_sync(all, rr, o);
    bb += __shfl_xor_sync(all, bb, o);
  }
  if (lane == 0) {
    sm[0][wp] = rr;
    sm[1][wp] = bb;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double s0 = 0.0, s1 = 0.0;
    for (int w = 0; w < kNaWarps; ++w) {
      s0 += sm[0][w];
      s1 += sm[1][w];
    }
    partials[2 * blockIdx.x] = s0;
    partials[2 * blockIdx.x + 1] = s1;
    __threadfence();
    const uint32_t ticket = atomicAdd(counter, 1u);
    amlast = opm::noalloc_is_last(ticket, base, gridDim.x);
    if (opm::noalloc_is_foreign(ticket, base, gridDim.x)) line->spoilt = tag;
  }
  __syncthreads();
  if (!amlast) return;
  __threadfence();
  // the last CTA: partials strided over the threads, then the butterflies
  double s0 = 0.0, s1 = 0.0;
#pragma unroll 8
  for (unsigned t = threadIdx.x; t < gridDim.x; t += kNaThreads) {
    s0 += __ldcg(partials + 2 * t);
    s1 += __ldcg(partials + 2 * t + 1);
  }
  for (int o = 16; o > 0; o >>= 1) {
    s0 += __shfl_xor_sync(all, s0, o);
    s1 += __shfl_xor_sync(all, s1, o);
  }
  if (lane == 0) {
    sm[0][wp] = s0;
    sm[1][wp] = s1;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  s0 = s1 = 0.0;
  for (int w = 0; w < kNaWarps; ++w) {
    s0 += sm[0][w];
    s1 += sm[1][w];
  }
  const bool faulty = __ldcg(bad) == tag;
  norms[0] = faulty ? nan("") : sqrt(s0);
  norms[1] = faulty ? nan("") : sqrt(s1);
  line->outcome = opm::noalloc_outcome(tag, faulty ? opm::kNoallocFault : opm::kNoallocDone);
}

opm::NoallocPage g_host_page;
bool g_host_registered = false;

// The address on the current device dev of its line, NULL when the page
// cannot be registered.
NoallocLine *line_address(int dev) {
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  if (!g_host_registered) {
    if (cudaHostRegister(&g_host_page, sizeof(g_host_page), cudaHostRegisterPortable | cudaHostRegisterMapped) !=
        cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    g_host_registered = true;
  }
  void *p = nullptr;
  if (cudaHostGetDevicePointer(&p, &g_host_page, 0) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return &static_cast<opm::NoallocPage *>(p)->line[dev];
}

}  // namespace

extern "C" opm_status opm_bsr_residual_noalloc(int32_t nb, const int32_t *rowptr, const int32_t *colidx,
                                               const double *vals, const double *x, const double *b,
                                               double *r, double *norms, void *stream) {
  if (nb < 0 || nb > kNaMaxRows) return OPM_ERR_ARG;  // beyond the scratch capacity
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return OPM_ERR_ARG;
  }
  if (!on_device(norms, dev)) return OPM_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (nb == 0) {
    if (cudaMemsetAsync(norms, 0, 2 * sizeof(double), st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
      cudaGetLastError();
      return OPM_ERR_CUDA;
    }
    return OPM_OK;
  }
  if (!on_device(rowptr, dev) || !on_device(colidx, dev) || !on_device(vals, dev) || !on_device(x, dev) ||
      !on_device(b, dev) || !on_device(r, dev))
    return OPM_ERR_ARG;
  unsigned char *scratch = nullptr;
  opm_status s = scratch_address(dev, &scratch);
  if (s != OPM_OK) return s;
  // as many CTAs as fit on the device at once: a CTA's sums end in 20 FP64
  // additions per warp, as much as the product of one group
  int sms = 1;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return OPM_ERR_CUDA;
  }
  const int tiles = std::min((nb + kNaTile - 1) / kNaTile, std::min(8 * sms, kNaMaxTiles));
  NoallocLine *line = line_address(dev);
  if (!line) return OPM_ERR_CUDA;
  NoallocCall call;
  {
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    call = g_calls[dev].begin((uint32_t)tiles);
  }
  bool ran = !call.clear || cudaMemsetAsync(scratch, 0, kNaCounterBytes, st) == cudaSuccess;
  if (ran) {
    k_residual_noalloc<<<tiles, kNaThreads, 0, st>>>(nb, rowptr, colidx, vals, x, b, r, norms, scratch, line,
                                                     call.base, call.tag);
    ran = cudaGetLastError() == cudaSuccess;
    ran = cudaStreamSynchronize(st) == cudaSuccess && ran;
  }
  const NoallocLine &out = g_host_page.line[dev];
  const uint64_t outcome = out.outcome;
  if (!ran || out.spoilt == call.tag || outcome >> 32 != call.tag) {
    cudaGetLastError();
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    g_calls[dev].unsure = true;
    return OPM_ERR_CUDA;
  }
  return (uint32_t)outcome == opm::kNoallocFault ? OPM_ERR_PATTERN : OPM_OK;
}
