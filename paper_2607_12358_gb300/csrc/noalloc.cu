// acid_drift_signal_noalloc: the drift reduction for callers that cannot
// allocate device memory at all, not even a workspace to hand to
// acid_drift_signal.  Examples: a plugin that only receives its input and
// output buffers from a host framework, or an inference process whose device
// memory is entirely reserved by another allocator.
//
// The reduction's scratch (one fp64 partial pair per thread block plus the
// three results) lives in the file-scope array below instead of a
// caller-provided workspace.  Every GPU that loads this library holds the
// array until the process exits.
#include <mutex>
#include <string>

#define ACID_UNIT_WITHOUT_WAITS
#include "common.cuh"
#include "internal.h"

namespace acid {

namespace {

constexpr size_t kNoAllocScratchBytes = 16 * 1024;
// Largest element count accepted.  The reduction runs a fixed grid of 608
// blocks of 256 threads, and each thread sums |cur - prev| and |prev| into
// two fp32 accumulators each, so at n = 2^31 an accumulator adds at most
// 2^31 / (608 * 256 * 2) < 6,900 terms.  Summing non-negative terms one by one
// in fp32 has a relative error of at most (terms - 1) * 2^-24 < 4.2e-4, and
// the fp64 stages after it add nothing at that scale, so the ratio of the two
// sums stays within about 8.4e-4 of exact even in the worst case: inside the
// 1e-3 drift tolerance.  (The expected error, which grows with the square
// root of the term count, is far smaller.)
constexpr int64_t kNoAllocMaxElems = int64_t(1) << 31;
constexpr int kMaxDevices = 64;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

std::mutex g_mu;
struct ScratchSlot {
  unsigned long long ctx;  // id of the context that the address belongs to
  void* addr;
};
ScratchSlot g_slot[kMaxDevices] = {};

// Device address of the scratch array in the current device's context (host
// code cannot use the symbol itself as a device pointer).  Looked up once per
// context: after cudaDeviceReset, which unloads the library's device code, the
// device's context has a new id, though its handle stays the same.
acid_status scratch_address(void** out) {
  int dev = 0;
  ACID_CUDA(cudaGetDevice(&dev));
  ACID_REQUIRE(dev >= 0 && dev < kMaxDevices, ACID_ERR_UNSUPPORTED, "drift_noalloc: device index too large");
  std::lock_guard<std::mutex> lk(g_mu);
  ScratchSlot& sl = g_slot[dev];
  const unsigned long long ctx = context_id();
  if (ctx == 0 || sl.ctx != ctx) {
    // the lookup also makes the device's context current, so its id is read after it
    ACID_CUDA(cudaGetSymbolAddress(&sl.addr, g_noalloc_scratch));
    sl.ctx = context_id();
  }
  *out = sl.addr;
  return ACID_OK;
}

}  // namespace
}  // namespace acid

using namespace acid;

extern "C" acid_status acid_drift_signal_noalloc(const void* prev, const void* cur, int64_t n, int32_t dtype,
                                                 double* out_rel_l1, double* out_sums, acid_stream_t stream) {
  clear_error();
  ACID_REQUIRE(dtype == ACID_BF16 || dtype == ACID_FP32, ACID_ERR_INVALID_ARG, "drift_noalloc: unknown dtype");
  ACID_REQUIRE(n >= 0, ACID_ERR_INVALID_ARG, "drift_noalloc: n must be >= 0");
  ACID_REQUIRE(n <= kNoAllocMaxElems, ACID_ERR_UNSUPPORTED,
               "drift_noalloc: n = " + std::to_string(n) + " exceeds the maximum of " +
                   std::to_string(kNoAllocMaxElems) + " elements; use acid_drift_signal with a workspace");
  ACID_REQUIRE(out_rel_l1 != nullptr, ACID_ERR_INVALID_ARG, "drift_noalloc: out_rel_l1 is null");
  ACID_REQUIRE(n == 0 || (prev && cur), ACID_ERR_INVALID_ARG, "drift_noalloc: null input");
  ACID_REQUIRE(n == 0 || (aligned(prev, 16) && aligned(cur, 16)), ACID_ERR_UNSUPPORTED,
               "drift_noalloc: inputs must be 16-byte aligned");
  const size_t part_bytes = drift_workspace_bytes(n);
  ACID_REQUIRE(part_bytes + 3 * sizeof(double) <= kNoAllocScratchBytes, ACID_ERR_UNSUPPORTED,
               "drift_noalloc: scratch array too small for this build");
  void* scratch = nullptr;
  ACID_TRY(scratch_address(&scratch));
  cudaStream_t s = (cudaStream_t)stream;
  double* result = reinterpret_cast<double*>(static_cast<uint8_t*>(scratch) + part_bytes);
  DriftOutputs outs(out_rel_l1, out_sums);
  // Every partial slot the final pass reads is written earlier in the same
  // call, and the results are overwritten, so nothing needs clearing here.
  if (n == 0) {
    outs.rel_direct = outs.sums_direct = nullptr;
    ACID_CUDA(cudaMemsetAsync(result, 0, 3 * sizeof(double), s));
  } else {
    ACID_TRY(drift_launch(dtype, prev, cur, nullptr, nullptr, n, result, scratch, part_bytes, s, outs.rel_direct,
                          outs.sums_direct));
  }
  return outs.finish(result, s);
}
