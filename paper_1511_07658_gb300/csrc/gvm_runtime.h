// Internal functions shared by the host runtime translation units.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "gvm.h"
#include "gvm_internal.h"

namespace gvm {

enum : int { kPathFma = 0, kPathSplit3 = 1 };

// Driver entry points, resolved once through the runtime (no link-time libcuda).
struct DriverApi {
  CUresult (*write_value32)(CUstream, CUdeviceptr, cuuint32_t, unsigned int);
  CUresult (*wait_value32)(CUstream, CUdeviceptr, cuuint32_t, unsigned int);
  CUresult (*encode_tiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                           const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                           CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
};
// Returns nullptr if the driver or an entry point is unavailable.
const DriverApi* driver_api();

// Tensor maps of a row-major binary32 A (m x k) and B (k x n) for the pair
// form. Rows of a multiple of 16 bytes from a 16-byte aligned base: boxes of
// 128 rows x 32 values (A) and 32 rows x 32 values (B), landing with the
// 128-byte swizzle. Otherwise the rows are mapped in fours (packed). Returns
// the kPrMap* / kPrPacked* bits (gvm_pair.cuh) of what could be mapped.
uint32_t encode_pair_maps(const float* A, const float* B, int32_t m, int64_t n, int32_t k, CUtensorMap* tmA,
                          CUtensorMap* tmB);

// Most columns of a pair-form tile whose operands have these maps.
int pair_tile_n(uint32_t maps);

// Scheduler kernel: the most CTAs the device (of `sms` SMs) holds at once on
// `path`, dynamic smem bytes, and an asynchronous launch on `stream` (the pair
// form's grid is a multiple of two).
cudaError_t scheduler_setup(int path, int sms, int* max_ctas, size_t* smem_bytes);
cudaError_t launch_scheduler(int path, const SchedParams& p, int grid, size_t smem, cudaStream_t stream);

// A manager's worker threads for the SPMD harnesses (gvm_spmd.cu): none until a
// run needs them, then kept for the next run and joined with the manager.
class WorkerPool;
WorkerPool* worker_pool_create();
void worker_pool_destroy(WorkerPool* pool);
WorkerPool* ctx_workers(gvm_ctx* ctx);

// Configuration of a manager, for the library's other host modules.
int ctx_mode(const gvm_ctx* ctx);
int ctx_max_ranks(const gvm_ctx* ctx);
// Counts the gvm_ipc servers using a manager (gvm_shutdown refuses while any is).
void ctx_servers_add(gvm_ctx* ctx, int delta);

}  // namespace gvm
