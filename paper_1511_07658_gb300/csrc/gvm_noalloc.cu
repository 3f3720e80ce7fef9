// gvm_sgemm_f32_noalloc: the split3 SGEMM task kernel for callers that
// cannot allocate device memory.
//
// The regular entry point's GVM_SGEMM_SPLIT3 takes scratch from the caller.
// Some callers have no way to provide it: a plain C program linking this
// library with no device allocator of its own, a framework whose memory pool
// already owns all device memory, or a latency-critical serving loop where
// allocating (and the device-wide synchronisation cudaFree implies) is not
// allowed. The kernel splits its operands while staging them, so none is
// needed; the shape bound is the entry point's documented one.
#include "gvm.h"
#include "gvm_internal.h"

namespace {

constexpr uint64_t kNoAllocScratchBytes = 32ull << 20;  // 4 (m + n) kp bytes: up to m = n = k = 2048

}  // namespace

extern "C" int gvm_sgemm_f32_noalloc(const float* A, const float* B, float* C, int32_t m, int32_t n, int32_t k,
                                     void* stream) {
  if (m <= 0 || n <= 0 || k <= 0 || !A || !B || !C) return GVM_EINVAL;
  if (gvm::split_scratch_bytes(m, n, k) > kNoAllocScratchBytes) return GVM_ENOMEM;
  return gvm_sgemm_f32(A, B, C, m, n, k, GVM_SGEMM_SPLIT3_FUSED, nullptr, 0, stream);
}
