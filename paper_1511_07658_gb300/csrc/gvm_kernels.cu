// The task kernels on their own: gvm_vadd_f32 and gvm_sgemm_f32 run one
// task's kernel on caller-given device buffers without the manager. They use
// the same tile functions as the scheduler, so a task computed here and the
// same task computed by the manager agree bit for bit.
#include <cuda_runtime.h>
#include <string.h>

#include <atomic>
#include <mutex>

#include "gvm.h"
#include "gvm_device.cuh"
#include "gvm_pair.cuh"
#include "gvm_runtime.h"

namespace gvm {

// Last error status of a standalone kernel (0 = ok); see gvm_kernel_status.
__device__ uint32_t g_kernel_status;

__global__ void __launch_bounds__(kThreads) vadd_kernel(const float* a, const float* b, float* c, int64_t n,
                                                        int64_t chunk) {
  const int64_t lo = (int64_t)blockIdx.x * chunk;
  if (lo >= n) return;
  vadd_range(a, b, c, lo, min(n, lo + chunk), threadIdx.x, kThreads);
}

__global__ void __launch_bounds__(kThreads) vmul_kernel(const float* a, const float* b, float* c, int64_t n,
                                                        int64_t chunk, int iters) {
  const int64_t lo = (int64_t)blockIdx.x * chunk;
  if (lo >= n) return;
  vmul_range(a, b, c, lo, min(n, lo + chunk), threadIdx.x, kThreads, iters);
}

__global__ void __launch_bounds__(kFmaThreads, 2) fma_sgemm_kernel(const float* A, const float* B, float* C, int m,
                                                                 int n, int k) {
  extern __shared__ uint8_t dyn_smem[];
  fma_tile(A, B, C, m, n, k, blockIdx.y, blockIdx.x, reinterpret_cast<FmaSmem*>(dyn_smem));
}

// Pair form: a persistent grid of clusters of two CTAs; cluster i takes tiles
// i, i + clusters, ... (row-major over the tile grid). Every role walks the
// same sequence. k-steps are numbered through: 65536^3 has 1.8 million for
// each of 76 clusters, far from the wrap of a 32-bit number.
struct PrStandShared {
  PrShared ps;
  uint32_t abort_flag, fail_where;
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPrThreads, 1)
    pr_sgemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, uint32_t maps,
                    const float* A, const float* B, float* C, int m, int n, int k, int tile_n, uint64_t timeout_ns) {
  extern __shared__ __align__(1024) uint8_t dyn_smem[];
  uint8_t* land = dyn_smem;
  uint8_t* stages = dyn_smem + kPrLand * kPrLandBytes;
  PrStandShared& sh = *reinterpret_cast<PrStandShared*>(dyn_smem + kPrRingBytes);
  if (threadIdx.x == 0) {
    sh.abort_flag = 0;
    sh.fail_where = 0;
  }
  PrShared* ps = &sh.ps;
  pr_init(ps);
  const int warp = threadIdx.x >> 5;
  const int tiles_n = (n + tile_n - 1) / tile_n;
  const int ntiles = ((m + kPrM - 1) / kPrM) * tiles_n;
  const int first = blockIdx.x >> 1, stride = gridDim.x >> 1;
  const uint32_t nkb = (uint32_t)((k + kTcBK - 1) / kTcBK);
  uint32_t it = 0, tile_no = 0;
  auto tile_at = [&](int i) { return pr_tile(A, B, C, m, n, k, i / tiles_n, i % tiles_n, tile_n, maps); };
  if (warp < kPrEpiWarps) {
    for (int i = first; i < ntiles; i += stride, ++tile_no)
      if (!pr_epilogue(tile_at(i), ps, tile_no, timeout_ns, &sh.abort_flag, &sh.fail_where)) break;
  } else if (warp < kPrMmaWarp) {
    for (int i = first; i < ntiles; i += stride, it += nkb)
      if (!pr_convert(tile_at(i), land, stages, ps, it, it, timeout_ns, &sh.abort_flag, &sh.fail_where)) break;
  } else if (warp == kPrMmaWarp) {
    if (ps->cta == 0 && elect_one()) {
      for (int i = first; i < ntiles; i += stride, it += nkb, ++tile_no)
        if (!pr_mma(tile_at(i), stages, ps, it, tile_no, timeout_ns, &sh.abort_flag, &sh.fail_where, nullptr)) break;
      umma_commit_pair(&ps->mma_done);
    }
    __syncwarp();
  } else if (warp == kPrProdWarp) {
    if (elect_one()) {
      uint32_t pend = 0;
      for (int i = first; i < ntiles; i += stride, it += nkb)
        if (!pr_produce(tile_at(i), land, ps, it, &tmA, &tmB, timeout_ns, &sh.abort_flag, &sh.fail_where, pend)) break;
      pr_produce_quiesce(ps, pend, timeout_ns);
    }
    __syncwarp();
  }
  pr_teardown(ps, 2 * timeout_ns);
  if (threadIdx.x == 0 && sh.abort_flag) atomicExch(&g_kernel_status, kStatusTimeout | (sh.fail_where << 8));
}

// ---------------------------------------------------------------- driver API

static DriverApi g_api;
static bool g_api_ok = false;
static std::once_flag g_api_once;

const DriverApi* driver_api() {
  std::call_once(g_api_once, [] {
    cudaDriverEntryPointQueryResult q;
    void* f1 = nullptr;
    void* f2 = nullptr;
    void* f3 = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuStreamWriteValue32", &f1, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return;
    if (cudaGetDriverEntryPointByVersion("cuStreamWaitValue32", &f2, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f3, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return;
    g_api.write_value32 = reinterpret_cast<decltype(g_api.write_value32)>(f1);
    g_api.wait_value32 = reinterpret_cast<decltype(g_api.wait_value32)>(f2);
    g_api.encode_tiled = reinterpret_cast<decltype(g_api.encode_tiled)>(f3);
    g_api_ok = true;
  });
  return g_api_ok ? &g_api : nullptr;
}

uint32_t encode_pair_maps(const float* A, const float* B, int32_t m, int64_t n, int32_t k, CUtensorMap* tmA,
                          CUtensorMap* tmB) {
  const DriverApi* api = driver_api();
  if (!api) return 0;
  // A rows x cols operand: bit `map` when it has a map, bit `packed` when its
  // rows are mapped in fours.
  auto encode = [&](const float* p, uint64_t rows, uint64_t cols, uint32_t box_rows, uint32_t pack_cols, CUtensorMap* tm,
                    uint32_t map, uint32_t packed) -> uint32_t {
    const uintptr_t base = reinterpret_cast<uintptr_t>(p);
    const bool pack = (cols % 4) != 0 || (base & 15) != 0;
    if (pack && rows < 4) return 0;
    const uint64_t shift = (base & 15) / 4;  // values between the aligned base and the operand
    const cuuint64_t dims[2] = {pack ? 4 * cols + shift : cols, pack ? rows / 4 : rows};
    const cuuint64_t strides[1] = {pack ? cols * 16 : cols * 4};
    const cuuint32_t box[2] = {pack ? pack_cols : 32u, pack ? box_rows / 4 : box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = api->encode_tiled(
        tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, reinterpret_cast<void*>(base & ~uintptr_t(15)), dims, strides, box, estr,
        CU_TENSOR_MAP_INTERLEAVE_NONE, pack ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_128B,
        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return 0;
    return map | (pack ? packed : 0u);
  };
  return encode(A, (uint64_t)m, (uint64_t)k, 128, kPrPackA, tmA, kPrMapA, kPrPackedA) |
         encode(B, (uint64_t)k, (uint64_t)n, 32, kPrPackB, tmB, kPrMapB, kPrPackedB);
}

int pair_tile_n(uint32_t maps) { return maps == (kPrMapA | kPrMapB) ? kPrN : kPrPackedN; }

constexpr uint64_t kStandaloneTimeoutNs = 10ull * 1000 * 1000 * 1000;

static int sm_count() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  }
  return sms;
}

}  // namespace gvm

using namespace gvm;

extern "C" int gvm_vadd_f32(const float* a, const float* b, float* c, int64_t n, void* stream) {
  if (n < 0) return GVM_EINVAL;
  if (n == 0) return GVM_OK;
  if (!a || !b || !c) return GVM_EINVAL;
  const int sms = sm_count();
  if (sms <= 0) return GVM_ENODEV;
  int64_t chunk = (n + (int64_t)sms * 4 - 1) / ((int64_t)sms * 4);
  chunk = (chunk + 1023) / 1024 * 1024;
  if (chunk < kVaddTileMin) chunk = kVaddTileMin;
  const int64_t grid = (n + chunk - 1) / chunk;
  vadd_kernel<<<(unsigned)grid, kThreads, 0, static_cast<cudaStream_t>(stream)>>>(a, b, c, n, chunk);
  return cudaGetLastError() == cudaSuccess ? GVM_OK : GVM_EDEVICE;
}

extern "C" int gvm_vmul_f32(const float* a, const float* b, float* c, int64_t n, int32_t iters, void* stream) {
  if (n < 0 || iters < 1 || iters > 1024) return GVM_EINVAL;
  if (n == 0) return GVM_OK;
  if (!a || !b || !c) return GVM_EINVAL;
  const int sms = sm_count();
  if (sms <= 0) return GVM_ENODEV;
  int64_t chunk = (n + (int64_t)sms * 4 - 1) / ((int64_t)sms * 4);
  chunk = (chunk + 1023) / 1024 * 1024;
  if (chunk < kVaddTileMin) chunk = kVaddTileMin;
  const int64_t grid = (n + chunk - 1) / chunk;
  vmul_kernel<<<(unsigned)grid, kThreads, 0, static_cast<cudaStream_t>(stream)>>>(a, b, c, n, chunk, iters);
  return cudaGetLastError() == cudaSuccess ? GVM_OK : GVM_EDEVICE;
}

extern "C" uint64_t gvm_sgemm_scratch_bytes(int32_t m, int32_t n, int32_t k, int32_t path) {
  if (m <= 0 || n <= 0 || k <= 0) return 0;
  return path == GVM_SGEMM_SPLIT3 ? split_scratch_bytes(m, n, k) : 0;
}

// The large-shared-memory attribute is set on every call, as for the
// scheduler: it belongs to the function in the current context, so a flag
// kept per process would skip it on a second device or after a reset.
template <typename F>
static int allow_smem(F* fn, size_t smem) {
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess
             ? GVM_OK
             : GVM_EDEVICE;
}

extern "C" int gvm_sgemm_f32(const float* A, const float* B, float* C, int32_t m, int32_t n, int32_t k,
                             int32_t path, void* scratch, uint64_t scratch_bytes, void* stream) {
  if (m <= 0 || n <= 0 || k <= 0 || m > 65536 || n > 65536 || k > 65536) return GVM_EINVAL;
  if (!A || !B || !C) return GVM_EINVAL;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (path == GVM_SGEMM_FMA) {
    const size_t smem = sizeof(FmaSmem);
    if (allow_smem(fma_sgemm_kernel, smem) != GVM_OK) return GVM_EDEVICE;
    dim3 grid((n + kFmaTile - 1) / kFmaTile, (m + kFmaTile - 1) / kFmaTile);
    fma_sgemm_kernel<<<grid, kFmaThreads, smem, s>>>(A, B, C, m, n, k);
    return cudaGetLastError() == cudaSuccess ? GVM_OK : GVM_EDEVICE;
  }
  // The split3 forms are one kernel; SPLIT3's scratch is still checked.
  if (path == GVM_SGEMM_SPLIT3) {
    if (!scratch || scratch_bytes < split_scratch_bytes(m, n, k) || (reinterpret_cast<uintptr_t>(scratch) & 255))
      return GVM_EINVAL;
  } else if (path != GVM_SGEMM_SPLIT3_FUSED && path != GVM_SGEMM_SPLIT3_WIDE) {
    return GVM_EINVAL;
  }
  const size_t smem = kPrRingBytes + sizeof(PrStandShared);
  if (allow_smem(pr_sgemm_kernel, smem) != GVM_OK) return GVM_EDEVICE;
  const int sms = sm_count();
  if (sms < 2) return GVM_ENODEV;
  const int pairs = sms / 2;
  // Columns per tile: the fewest waves of tiles weighted by a tile's time. A
  // k-step of 256 x n costs about 256 + n units (A's share of the staging
  // does not shrink with n). Measured, one launch from a cold L2, at 64 / 128 /
  // 192 / 256 columns: 512^3 16.4 / 16.4 / 18.4 / 20.5 us (64 taken), 2048^3
  // 107 / 64 / 68 / 43 (256 taken). Packed operands, 64 / 128 / 192: 1530 x 1027
  // x 2001 94 / 61 / 68 (128 taken), 2047^3 168 / 104 / 115 (128), 4095^3 1077 /
  // 584 / 487 (192).
  CUtensorMap tmA, tmB;
  memset(&tmA, 0, sizeof(tmA));
  memset(&tmB, 0, sizeof(tmB));
  const uint32_t maps = encode_pair_maps(A, B, m, n, k, &tmA, &tmB);
  int tile_n = 64;
  int64_t best = INT64_MAX;
  const int64_t rows = (m + kPrM - 1) / kPrM;
  for (int tn = pair_tile_n(maps); tn >= 64; tn -= 64) {
    const int64_t cost = (rows * ((n + tn - 1) / tn) + pairs - 1) / pairs * (256 + tn);
    if (cost < best) {
      best = cost;
      tile_n = tn;
    }
  }
  const int64_t tiles = rows * ((n + tile_n - 1) / tile_n);
  const int grid = 2 * (int)(tiles < pairs ? tiles : pairs);
  pr_sgemm_kernel<<<grid, kPrThreads, smem, s>>>(tmA, tmB, maps, A, B, C, m, n, k, tile_n, kStandaloneTimeoutNs);
  return cudaGetLastError() == cudaSuccess ? GVM_OK : GVM_EDEVICE;
}

// Reads and clears the error status of the standalone kernels (0 = ok; else
// low byte = status, next byte = which wait). Synchronous.
extern "C" int gvm_kernel_status(uint32_t* out) {
  if (!out) return GVM_EINVAL;
  uint32_t v = 0;
  if (cudaMemcpyFromSymbol(&v, g_kernel_status, sizeof(v)) != cudaSuccess) return GVM_EDEVICE;
  const uint32_t zero = 0;
  if (cudaMemcpyToSymbol(g_kernel_status, &zero, sizeof(zero)) != cudaSuccess) return GVM_EDEVICE;
  *out = v;
  return GVM_OK;
}
