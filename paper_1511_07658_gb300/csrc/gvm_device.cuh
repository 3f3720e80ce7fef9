// Device code shared by the persistent scheduler and the standalone task
// kernels: PTX wrappers, and one function per tile kind.
//
//   vadd_range   vector-add task (Table 2, VecAdd): c = a + b, binary32
//   vmul_range   vector-multiply task (Table 2, VecMul): iterated binary32 products
//   fma_tile     matrix-multiply task (Table 2, MM) on the CUDA cores
//
// Every wait is bounded by a deadline on %globaltimer; a wait that runs out
// reports failure to its caller, which records a status word and stops.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "gvm_internal.h"

namespace gvm {

// ---------------------------------------------------------------- PTX basics

__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint32_t ld_acquire_gpu(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint64_t ld_acquire_gpu64(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_acquire_sys(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.sys.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_relaxed_gpu(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint64_t ld_relaxed_gpu64(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_gpu(uint32_t* p, uint32_t v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void st_release_gpu64(uint64_t* p, uint64_t v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void st_release_sys(uint32_t* p, uint32_t v) {
  asm volatile("st.release.sys.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void st_relaxed_sys64(uint64_t* p, uint64_t v) {
  asm volatile("st.relaxed.sys.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
// 16-byte load that bypasses L1 (data written by other CTAs or by the host).
__device__ __forceinline__ uint4 ld_cg_v4(const void* p) {
  uint4 v;
  asm volatile("ld.global.cg.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p)
               : "memory");
  return v;
}
__device__ __forceinline__ uint4 ld_volatile_v4(const void* p) {
  uint4 v;
  asm volatile("ld.volatile.global.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p)
               : "memory");
  return v;
}
__device__ __forceinline__ void st_cg_v4(void* p, uint4 v) {
  asm volatile("st.global.cg.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z),
               "r"(v.w)
               : "memory");
}

__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}
__device__ __forceinline__ void fence_tensormap_release() {
  asm volatile("fence.proxy.tensormap::generic.release.gpu;" ::: "memory");
}
__device__ __forceinline__ void fence_tensormap_acquire(const void* tmap) {
  asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(tmap) : "memory");
}

// ---------------------------------------------------------------- mbarrier

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait for the phase with the given parity. Gives up when the
// deadline passes or another warp of the CTA has flagged an abort.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint64_t timeout_ns,
                                          volatile uint32_t* cta_abort) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t deadline = globaltimer() + timeout_ns;
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*cta_abort) return false;
    if (globaltimer() > deadline) return false;
  }
}

// ---------------------------------------------------------------- TMA

__device__ __forceinline__ void tma_load_2d(uint32_t smem_dst, const CUtensorMap* tm, int c0, int c1, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_dst),
      "l"(tm), "r"(c0), "r"(c1), "r"(smem_u32(bar))
      : "memory");
}

// ---------------------------------------------------------------- tcgen05

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// 32 lanes x 32 consecutive fp32 columns: thread t of the warp gets lane (base + t).
__device__ __forceinline__ void tmem_ld_32x32b_x32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
        "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
        "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major operand, 64-byte swizzle, rows of
// kTcBK bf16 (64 bytes), 8-row core groups 512 bytes apart.
__device__ __forceinline__ uint64_t sdesc_k64b(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);  // start address
  d |= (uint64_t)1 << 16;                    // leading byte offset (unused when swizzled)
  d |= (uint64_t)(512u >> 4) << 32;          // stride byte offset: 8 rows x 64 B
  d |= (uint64_t)1 << 46;                    // descriptor version
  d |= (uint64_t)4 << 61;                    // swizzle mode: 64 B
  return d;
}

// Instruction descriptor, kind::f16: D fp32, A and B bf16, both K-major, M x N.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// ---------------------------------------------------------------- vector add

// Elementwise tasks over [lo, hi), by threads tid = 0 .. nthr-1 (a CTA's
// share of one tile): float4 streaming loads (evict-first), 4 in flight per
// thread, scalar head/tail when the operands are not 16-byte aligned there.
//   ELEM_ADD: c[i] = a[i] + b[i]                     (Table 2, VecAdd)
//   ELEM_MUL: c[i] = (...((a[i] * b[i]) * b[i])...) * b[i], `iters` products
//             (Table 2, VecMul: 15 iterations), each rounded to nearest
enum : int { kElemAdd = 0, kElemMul = 1 };

// Two binary32 operations in one instruction, each rounded as __fmaf_rn /
// __fmul_rn would.
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
template <int OP>
__device__ __forceinline__ float elem_op(float x, float y, int iters) {
  if (OP == kElemAdd) return __fadd_rn(x, y);
  float z = x;
  for (int i = 0; i < iters; ++i) z = __fmul_rn(z, y);
  return z;
}

// Four elements: the products two at a time.
template <int OP>
__device__ __forceinline__ float4 elem_op4(const float4& x, const float4& y, int iters) {
  if (OP == kElemAdd)
    return make_float4(__fadd_rn(x.x, y.x), __fadd_rn(x.y, y.y), __fadd_rn(x.z, y.z), __fadd_rn(x.w, y.w));
  uint64_t z0 = pack2(x.x, x.y), z1 = pack2(x.z, x.w);
  const uint64_t y0 = pack2(y.x, y.y), y1 = pack2(y.z, y.w);
#pragma unroll 4
  for (int i = 0; i < iters; ++i) {
    z0 = mul2(z0, y0);
    z1 = mul2(z1, y1);
  }
  return make_float4(__uint_as_float((uint32_t)z0), __uint_as_float((uint32_t)(z0 >> 32)), __uint_as_float((uint32_t)z1),
                     __uint_as_float((uint32_t)(z1 >> 32)));
}

// kL2: operands are read past L1 (ld.global.cg). Needed where a CTA learns of
// the task from another SM (the pair scheduler's peer CTA): its own L1 may
// still hold an earlier task's values of the same staging addresses.
template <bool kL2>
__device__ __forceinline__ float4 ld_stream(const float4* p) {
  return kL2 ? __ldcg(p) : __ldcs(p);
}
template <bool kL2>
__device__ __forceinline__ float ld_stream(const float* p) {
  return kL2 ? __ldcg(p) : *p;
}

template <int OP, bool kL2>
__device__ __forceinline__ void elementwise_range(const float* __restrict__ a, const float* __restrict__ b,
                                                  float* __restrict__ c, int64_t lo, int64_t hi, int tid, int nthr,
                                                  int iters) {
  const bool vec = ((reinterpret_cast<uintptr_t>(a + lo) | reinterpret_cast<uintptr_t>(b + lo) |
                     reinterpret_cast<uintptr_t>(c + lo)) &
                    15) == 0;
  int64_t done = lo;
  if (vec) {
    constexpr int U = 4;  // loads of each operand in flight a thread
    const int64_t nv = (hi - lo) >> 2;
    const float4* a4 = reinterpret_cast<const float4*>(a + lo);
    const float4* b4 = reinterpret_cast<const float4*>(b + lo);
    float4* c4 = reinterpret_cast<float4*>(c + lo);
    int64_t i = tid;
    for (; i + (int64_t)(U - 1) * nthr < nv; i += (int64_t)U * nthr) {
      float4 x[U], y[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        x[u] = ld_stream<kL2>(a4 + i + u * nthr);
        y[u] = ld_stream<kL2>(b4 + i + u * nthr);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) __stcs(c4 + i + u * nthr, elem_op4<OP>(x[u], y[u], iters));
    }
    for (; i < nv; i += nthr)
      __stcs(c4 + i, elem_op4<OP>(ld_stream<kL2>(a4 + i), ld_stream<kL2>(b4 + i), iters));
    done = lo + (nv << 2);
  }
  for (int64_t i = done + tid; i < hi; i += nthr) c[i] = elem_op<OP>(ld_stream<kL2>(a + i), ld_stream<kL2>(b + i), iters);
}

template <bool kL2 = false>
__device__ __forceinline__ void vadd_range(const float* __restrict__ a, const float* __restrict__ b,
                                           float* __restrict__ c, int64_t lo, int64_t hi, int tid, int nthr) {
  elementwise_range<kElemAdd, kL2>(a, b, c, lo, hi, tid, nthr, 0);
}
template <bool kL2 = false>
__device__ __forceinline__ void vmul_range(const float* __restrict__ a, const float* __restrict__ b,
                                           float* __restrict__ c, int64_t lo, int64_t hi, int tid, int nthr,
                                           int iters) {
  elementwise_range<kElemMul, kL2>(a, b, c, lo, hi, tid, nthr, iters);
}

// ---------------------------------------------------------------- FMA SGEMM

struct FmaSmem {
  float As[2][kFmaBK][kFmaTile + 4];  // k-major copy of the A panel
  float Bs[2][kFmaBK][kFmaTile + 4];
};

// One 128 x 128 tile (tm, tn) of C = A B in binary32 FMA, by kFmaThreads = 128
// threads of 16 x 8 outputs. Every output accumulates k = 0, 1, ..., K-1 in
// order in one register. What bounds it is shared-memory reads against FMA
// issue: a 16-byte read takes 4 wavefronts whatever its lanes share, so a
// k step of an 8 x 8 thread tile costs 16 wavefronts for 64 FMA a lane, one of
// 16 x 8 24 for 128; two FMAs an instruction (fma.rn.f32x2) leave issue slots
// for the reads.
__device__ __forceinline__ void fma_tile(const float* __restrict__ A, const float* __restrict__ B,
                                         float* __restrict__ C, int m, int n, int k, int tm, int tn,
                                         FmaSmem* s) {
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const int row0 = tm * kFmaTile, col0 = tn * kFmaTile;
  const bool vec = ((k & 3) == 0) && ((n & 3) == 0) &&
                   ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15) == 0;
  const int lb_k = tid >> 3, lb_c = (tid & 7) * 4;  // B panel: k, first column (then every 32nd)
  float ra[16], rb[16];

  // A panel: row tid, 16 values of k. Elements outside A and B are zero.
  auto load = [&](int kt) {
    const int kb = kt * kFmaBK;
    const int r = row0 + tid, bk = kb + lb_k;
    const float* pa = A + (int64_t)r * k + kb;
    const float* pb = B + (int64_t)bk * n + col0 + lb_c;
    if (vec) {
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f), w = v;
        if (r < m && kb + 4 * h < k) v = *reinterpret_cast<const float4*>(pa + 4 * h);
        if (bk < k && col0 + lb_c + 32 * h < n) w = *reinterpret_cast<const float4*>(pb + 32 * h);
        ra[4 * h + 0] = v.x; ra[4 * h + 1] = v.y; ra[4 * h + 2] = v.z; ra[4 * h + 3] = v.w;
        rb[4 * h + 0] = w.x; rb[4 * h + 1] = w.y; rb[4 * h + 2] = w.z; rb[4 * h + 3] = w.w;
      }
    } else {
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        ra[i] = (r < m && kb + i < k) ? pa[i] : 0.f;
        const int c = (i & 3) + 32 * (i >> 2);
        rb[i] = (bk < k && col0 + lb_c + c < n) ? pb[c] : 0.f;
      }
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int i = 0; i < 16; ++i) s->As[buf][i][tid] = ra[i];
#pragma unroll
    for (int h = 0; h < 4; ++h)
      *reinterpret_cast<float4*>(&s->Bs[buf][lb_k][lb_c + 32 * h]) =
          make_float4(rb[4 * h], rb[4 * h + 1], rb[4 * h + 2], rb[4 * h + 3]);
  };

  // Rows 32 (i / 4) + 4 ty + i % 4; columns 64 (j / 2) + 4 tx + 2 (j % 2) and the next.
  uint64_t acc[16][4];
#pragma unroll
  for (int i = 0; i < 16; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0;

  const int nkt = (k + kFmaBK - 1) / kFmaBK;
  load(0);
  store(0);
  __syncthreads();
  for (int kt = 0; kt < nkt; ++kt) {
    const int buf = kt & 1;
    if (kt + 1 < nkt) load(kt + 1);
#pragma unroll
    for (int kk = 0; kk < kFmaBK; ++kk) {
      float av[16];
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const float4 a = *reinterpret_cast<const float4*>(&s->As[buf][kk][32 * h + ty * 4]);
        av[4 * h] = a.x; av[4 * h + 1] = a.y; av[4 * h + 2] = a.z; av[4 * h + 3] = a.w;
      }
      const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(&s->Bs[buf][kk][tx * 4]);
      const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(&s->Bs[buf][kk][64 + tx * 4]);
      const uint64_t bv[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const uint64_t aa = pack2(av[i], av[i]);
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma2(aa, bv[j], acc[i][j]);
      }
    }
    if (kt + 1 < nkt) store(buf ^ 1);
    __syncthreads();
  }

  const bool cvec = ((n & 3) == 0) && ((reinterpret_cast<uintptr_t>(C) & 15) == 0);
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int r = row0 + 32 * (i >> 2) + ty * 4 + (i & 3);
    if (r >= m) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = col0 + h * 64 + tx * 4;
      float* dst = C + (int64_t)r * n + c;
      if (cvec && c + 3 < n) {
        *reinterpret_cast<ulonglong2*>(dst) = make_ulonglong2(acc[i][2 * h], acc[i][2 * h + 1]);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (c + j < n) dst[j] = __uint_as_float((uint32_t)(acc[i][2 * h + (j >> 1)] >> (32 * (j & 1))));
      }
    }
  }
}

}  // namespace gvm
