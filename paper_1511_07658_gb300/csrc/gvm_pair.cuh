// Split3 SGEMM on CTA pairs ("pair form"): 256 x 256 tiles of a cluster of
// two CTAs, two-SM tensor-core MMAs (tcgen05 cta_group::2), binary32 operands
// landed by tensor copies and split from a landing ring into a bf16 ring.
//
// What bounds a split3 tile is shared memory: per k-step of 32, a CTA writes
// the landed binary32 operands, reads them, writes the bf16 planes and the
// tensor core reads them six times. On one CTA with a 128 x 256 tile that is
// 48 + 48 + 48 + 72 KB, 1728 clocks at 128 B a clock for 768 clocks of MMA. A
// pair shares the B operand between its two SMs (each stages 128 of the 256
// columns, the MMA reads both halves), so each CTA moves 32 + 32 + 32 + 48 KB,
// 1152 clocks for the same 768, and draws two thirds of the bytes from L2.
//
// The landing ring (kPrLand stages) holds only operands in flight and is
// released as soon as the converting warps have read it into registers, so
// up to 128 KB a CTA is on its way from L2 without holding registers; the
// bf16 ring (kPrStages) decouples the conversion from the MMAs. Aligned
// operands are read into registers before the stage is awaited. With three
// landings of 35 KB and the stage awaited first, 1024 products of 512^3 took
// 0.80 ms (now 0.74), the grouped mix 2.23 (2.01), 2048^3 43 us (39) and 64
// vector adds of 4 M values 0.55 ms (0.50).
//
// CTA roles (kPrThreads = 480, one CTA per SM):
//   warps 0-3    epilogue: TMEM lanes 32 w .. +31 of a finished accumulator
//                into C, while the next tile's MMAs fill the other one;
//   warps 4-11   converters, two groups of four warps taking alternate k-steps;
//   warp 12      MMA issue (one thread, in the even CTA -- the leader -- only);
//   warp 13      the scheduler's tile claims (leader) and their slots' return (peer);
//   warp 14      producer: one thread issues the tensor copies.
// The single threads are elected with elect.sync: the compiler then keeps
// their operands in uniform registers. Picked by lane == 0, an MMA took 133
// clocks to issue (elected: 54) and a k-step's five tensor copies 480 (271).
//
// Landing of an operand whose rows are multiples of 16 bytes (aligned): A, the
// CTA's 128 rows x 32 values as 128-byte rows, one box; B, up to four slabs of
// 32 k-rows x 32 columns (128-byte rows, 4 KB a slab), a box each. 16-byte
// chunk j of row r lies at chunk j ^ (r % 8) (the copies' 128-byte swizzle), so
// a warp's reads of 8 rows hit every bank once.
//
// Other row lengths (packed): a tensor copy wants row pitches and starts that
// are multiples of 16 bytes. Four consecutive rows of k values are one row of
// 4 k values whose pitch is such a multiple, so the matrix is mapped in rows
// of four ("super-rows"), and row 4 i + j is fetched from super-row i at value
// j k + kk, rounded down to a multiple of 4: boxes of 36 values (A) or 100 (B),
// one per j, whose first d_j = (j k) % 4 values are skipped when read. With k
// odd the four d_j differ, and the 4-byte reads of a warp (8 rows x 4 groups
// of 8 values) fall on 32 different banks. Rows beyond the last whole
// super-row (at most three) and what has no map are read from global memory
// by the converters. Before, such operands were loaded by 4-byte loads, 8 rows
// apart a lane: 1530 x 1027 x 2001 took 200 us on 128 x 256 tiles.
//
// bf16 stage (32 KB): A hi, A lo [128 rows][32 k] K-major; B hi, B lo
// [32 k][128 n] MN-major; 64-byte swizzle on atoms of 8 rows x 64 bytes (B
// atom (g, b): k rows 8g..+7, columns 32b..+31, at 2048 g + 512 b).
//
// A tile's column count is a multiple of 64 up to kPrN: the last column of
// tiles, and tiles of a product too small to fill the GPU, run MMAs of 64,
// 128 or 192 columns instead of padding to 256.
//
// Order of accumulation per element: k in steps of 16, AlBh, AhBl, AhBh each,
// as in every split3 form: bitwise the same results.
#pragma once

#include "gvm_device.cuh"
#include "gvm_ring.h"

namespace gvm {

constexpr int kPrM = 256;  // rows of a pair tile (128 per CTA)
constexpr int kPrN = 256;  // most columns of a pair tile (half per CTA)
// Four landings and three stages. Barriers of landings and stages always belong
// to the same converter group: landing q % 4's, and for the stages six, q % 6.
// (A group meets stage q % 3 at every second use only; at a barrier of the
// stage's own it would wait for the same parity each time, and a parity does
// not tell a phase from the one two before it.)
constexpr int kPrLand = 4;
static_assert(kPrLand % 2 == 0 && kPrBars % 2 == 0, "a group sees every phase of its barriers");
// Packed operands take more room in a landing, so that tiles with one have
// at most kPrPackedN columns.
constexpr int kPrPackedN = 192;
constexpr uint32_t kPrPackA = 36;                              // values a packed A row lands with
constexpr uint32_t kPrPackB = kPrPackedN / 2 + 4;              // values a packed B row lands with
constexpr uint32_t kPrSlab = 32 * 128;                         // one aligned slab: 32 k-rows x 32 columns
constexpr uint32_t kPrLandBytes = 32768;
constexpr uint32_t kPrLandA = 128 * 128, kPrLandPackA = 128 * kPrPackA * 4;  // A's bytes; B's landing follows
static_assert(kPrLandA + 4 * kPrSlab <= kPrLandBytes && kPrLandPackA + 32 * kPrPackB * 4 <= kPrLandBytes &&
                  kPrLandPackA + (kPrPackedN / 64) * kPrSlab <= kPrLandBytes && kPrLandPackA % 1024 == 0,
              "every mix of landings fits");
constexpr uint32_t kPrAOff = 0;                                // bf16 planes
constexpr uint32_t kPrAlOff = 128 * 64;
constexpr uint32_t kPrBOff = 2 * 128 * 64;
constexpr uint32_t kPrBlOff = kPrBOff + 128 * 64;
constexpr uint32_t kPrStageBytes = kPrBlOff + 128 * 64;        // 32 KB
constexpr uint32_t kPrBAtomN = 512;
constexpr uint32_t kPrBAtomK = 2048;
constexpr uint32_t kPrRingBytes = kPrLand * kPrLandBytes + kPrStages * kPrStageBytes;

constexpr int kPrEpiWarps = 4;
constexpr int kPrConvWarp0 = 4;
constexpr int kPrConvWarps = 8;
constexpr int kPrGroupWarps = 4;
constexpr int kPrMmaWarp = 12;
constexpr int kPrCtlWarp = 13;
constexpr int kPrProdWarp = 14;
constexpr int kPrThreads = 15 * 32;
constexpr int kPrTmemCols = 512;  // two accumulators of 128 lanes x 256 columns per CTA

struct PrShared {
  uint64_t landed[kPrLand];     // producer -> converters (one arrival + the copies' bytes)
  uint64_t land_free[kPrLand];  // converters (4 warps of the k-step's group) -> producer
  uint64_t full[kPrStages];     // leader: converters of both CTAs -> MMA (4 + 4 warps)
  uint64_t empty[kPrBars];      // both: MMA commit -> converters
  uint64_t acc_full[2];         // both: MMA commit -> epilogue
  uint64_t acc_empty[2];        // leader: epilogue warps of both CTAs -> MMA
  uint64_t mma_done;            // both: the last commit, before teardown
  uint32_t tmem_base;
  uint32_t cta;                 // rank in the pair, 0 = leader
};

// How an operand lands (PrTile::land bits).
enum : uint32_t { kPrMapA = 1u, kPrMapB = 2u, kPrPackedA = 4u, kPrPackedB = 8u };

// One pair tile as every role sees it; passed by value, so that it lives in
// registers (behind a reference it lay in local memory, read back from L2 in
// every k-step once the control warp's acquires had invalidated L1). ncols: columns of the MMA, a multiple
// of 64; row0, col0: first row and column; land: kPr* bits.
struct PrTile {
  const float* A;
  const float* B;
  float* C;
  int64_t n;
  int m;
  int k;
  int row0;
  int ncols;
  int64_t col0;
  uint32_t land;
};

__device__ __forceinline__ PrTile pr_tile(const float* A, const float* B, float* C, int m, int64_t n, int k, int tm,
                                          int tn, int tile_n, uint32_t land) {
  PrTile t{A, B, C, n, m, k, tm * kPrM, 0, (int64_t)tn * tile_n, land};
  const int64_t left = n - t.col0;
  t.ncols = left >= tile_n ? tile_n : (int)((left + 63) / 64 * 64);
  return t;
}

// ---------------------------------------------------------------- PTX, splitting

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint4 v) {
  asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}
__device__ __forceinline__ uint4 ld_shared_v4(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}
// Makes this thread's generic-proxy shared-memory stores visible to the
// async proxy (the tensor core reads the stage through it).
__device__ __forceinline__ void fence_proxy_async_shared() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ uint32_t swz64(uint32_t row, uint32_t chunk) {
  return row * 64u + ((chunk ^ ((row >> 1) & 3u)) << 4);
}

// x = hi + lo + r with hi = RN_bf16(x), lo = RN_bf16(x - hi), for 8 values; the
// residual x - hi (exact in binary32) is taken two at a time (sub.rn.f32x2).
// The bf16 pair packs element 2i in its low half, so its binary32 value is
// the half shifted up, and element 2i+1's is the high half with the low bits
// cleared.
__device__ __forceinline__ void split8_x2(const float (&v)[8], uint4& hi, uint4& lo) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __nv_bfloat162 hb = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    const uint32_t hu = *reinterpret_cast<const uint32_t*>(&hb);
    const float h0 = __uint_as_float(hu << 16), h1 = __uint_as_float(hu & 0xffff0000u);
    float d0, d1;
    asm("{\n\t.reg .b64 x, y, d;\n\t"
        "mov.b64 x, {%2, %3};\n\t"
        "mov.b64 y, {%4, %5};\n\t"
        "sub.rn.f32x2 d, x, y;\n\t"
        "mov.b64 {%0, %1}, d;\n\t}"
        : "=f"(d0), "=f"(d1)
        : "f"(v[2 * i]), "f"(v[2 * i + 1]), "f"(h0), "f"(h1));
    const __nv_bfloat162 lb = __floats2bfloat162_rn(d0, d1);
    h[i] = hu;
    l[i] = *reinterpret_cast<const uint32_t*>(&lb);
  }
  hi = make_uint4(h[0], h[1], h[2], h[3]);
  lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// 32-byte store of 8 floats; the address must be 32-byte aligned.
__device__ __forceinline__ void st_v8(float* p, const uint32_t* r) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(r[0]), "r"(r[1]), "r"(r[2]),
               "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}


__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Shared::cluster address of the same shared-memory location in CTA `rank`.
__device__ __forceinline__ uint32_t mapa_shared(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
// Arrives on the barrier at `bar`'s offset in CTA `rank` of the cluster,
// ordering this CTA's own accesses only (CTA-scope release): what the waiter
// goes on to do is issue MMAs, which read each CTA's shared memory in place. A
// cluster-scope release would also wait for all of the thread's earlier
// accesses to be performed cluster-wide: about 1000 clocks a k-step.
__device__ __forceinline__ void mbar_arrive_cta(uint64_t* bar, uint32_t rank) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(mapa_shared(smem_u32(bar), rank)) : "memory");
}
// The same with a cluster-scope release: the waiter in CTA `rank` reads what
// this thread wrote into that CTA's shared memory.
__device__ __forceinline__ void mbar_arrive_release_cta(uint64_t* bar, uint32_t rank) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(mapa_shared(smem_u32(bar), rank))
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait with cluster-scope acquire (arrivals from the other CTA).
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity, uint64_t timeout_ns,
                                                  volatile uint32_t* cta_abort) {
  if (mbar_try_wait_cluster(bar, parity)) return true;
  const uint64_t deadline = globaltimer() + timeout_ns;
  while (true) {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    if (*cta_abort) return false;
    if (globaltimer() > deadline) return false;
  }
}
// The same waits by all lanes of a converged warp, left by all of them
// together: what follows may be warp-collective (tcgen05.ld, shuffles). The
// limit comes by reference, to be read once a wait goes on and not held through
// the converters' loops.
template <bool kCluster>
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, const uint64_t& timeout_ns,
                                               volatile uint32_t* cta_abort) {
  auto done = [&]() -> bool {
    const bool ok = kCluster ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity);
    return __all_sync(0xffffffffu, ok) != 0;
  };
  if (done()) return true;
  const uint64_t deadline = globaltimer() + timeout_ns;
  while (true) {
    if (done()) return true;
    if (__any_sync(0xffffffffu, *cta_abort != 0 || globaltimer() > deadline)) return false;
  }
}
// Whole-cluster barrier; every thread of both CTAs must reach it.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void st_cluster_u32(uint32_t cluster_addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}
__device__ __forceinline__ void st_cluster_v4(uint32_t cluster_addr, uint4 v) {
  asm volatile("st.shared::cluster.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(cluster_addr), "r"(v.x), "r"(v.y), "r"(v.z),
               "r"(v.w)
               : "memory");
}
// True in one thread of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
  return r != 0;
}

__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                               uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives on `bar` (same offset) in both CTAs once the MMAs issued so far are done.
__device__ __forceinline__ void umma_commit_pair(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ uint64_t pr_desc_b(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(kPrBAtomN >> 4) << 16;
  d |= (uint64_t)(kPrBAtomK >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}

// ---------------------------------------------------------------- set-up

// Both CTAs: barriers, TMEM of the pair, then a cluster barrier so that no
// CTA arrives on the other's barriers before they exist.
__device__ __forceinline__ void pr_init(PrShared* ps) {
  if (threadIdx.x == 0) {
    ps->cta = cluster_ctarank();
    for (int i = 0; i < kPrLand; ++i) {
      mbar_init(&ps->landed[i], 1);
      mbar_init(&ps->land_free[i], kPrGroupWarps);
    }
    for (uint32_t i = 0; i < kPrBars; ++i) mbar_init(&ps->empty[i], 1);
    for (uint32_t s = 0; s < kPrStages; ++s) mbar_init(&ps->full[s], 2 * kPrGroupWarps);
    for (int b = 0; b < 2; ++b) {
      mbar_init(&ps->acc_full[b], 1);
      mbar_init(&ps->acc_empty[b], 2 * kPrEpiWarps);
    }
    mbar_init(&ps->mma_done, 1);
    mbar_fence_init();
  }
  if ((threadIdx.x >> 5) == kPrMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ps->tmem_base)),
                 "r"(kPrTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  tc_fence_after();
}

// Both CTAs, every thread, once all roles have stopped (the leader's MMA
// thread has committed to mma_done): free the pair's TMEM. Every MMA is done
// and every commit has arrived (bounded), and no CTA leaves while the other
// may still read its shared memory or arrive on its barriers.
__device__ __forceinline__ void pr_teardown(PrShared* ps, uint64_t timeout_ns) {
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile uint32_t never = 0;
    (void)mbar_wait(&ps->mma_done, 0, timeout_ns, &never);
  }
  __syncwarp();
  cluster_sync();
  tc_fence_after();
  if ((threadIdx.x >> 5) == kPrMmaWarp)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(ps->tmem_base), "r"(kPrTmemCols)
                 : "memory");
}

// A wait of this CTA ran out: stop its other roles and the peer's.
__device__ __forceinline__ void pr_fail(PrShared* ps, uint32_t* cta_abort, uint32_t* fail_where, uint32_t where) {
  *fail_where = where;
  *reinterpret_cast<volatile uint32_t*>(cta_abort) = 1;
  st_cluster_u32(mapa_shared(smem_u32(cta_abort), ps->cta ^ 1u), 1);
}

// ---------------------------------------------------------------- producer

// Values of an operand before its 16-byte aligned base.
__device__ __forceinline__ uint32_t pr_shift(const float* p) {
  return (uint32_t)(reinterpret_cast<uintptr_t>(p) >> 2) & 3u;
}

// The producer thread: the tensor copies of every k-step of tile t, each
// k-step once the converters have read what its landing held. pend: bit 2i =
// a copy was issued into landing i, bit 2i + 1 = the parity of its phase.
// Returns false when a wait ran out.
__device__ __forceinline__ bool pr_produce(const PrTile t, uint8_t* land, PrShared* ps, uint32_t it,
                                           const CUtensorMap* tmA, const CUtensorMap* tmB, uint64_t timeout_ns,
                                           uint32_t* cta_abort, uint32_t* fail_where, uint32_t& pend) {
  const int nkb = (t.k + kTcBK - 1) / kTcBK;
  const uint32_t cta = ps->cta;
  const int row0 = t.row0 + (int)cta * 128;
  const int slabs = t.ncols >> 6;  // 32-column slabs of this CTA
  const int col0 = (int)t.col0 + (int)cta * (t.ncols >> 1);
  const bool map_a = (t.land & kPrMapA) != 0 && row0 < t.m, map_b = (t.land & kPrMapB) != 0;
  const bool pack_a = (t.land & kPrPackedA) != 0, pack_b = (t.land & kPrPackedB) != 0;
  const uint32_t tx = (map_a ? (pack_a ? 128u * kPrPackA * 4u : 128u * 128u) : 0u) +
                      (map_b ? (pack_b ? 32u * kPrPackB * 4u : (uint32_t)slabs * kPrSlab) : 0u);
  const uint32_t land0 = smem_u32(land);
  const int xa = (int)pr_shift(t.A), xb = (int)pr_shift(t.B) + col0, n = (int)t.n;
  for (int kb = 0; kb < nkb; ++kb) {
    const uint32_t q = it + (uint32_t)kb, i = q % kPrLand;
    if (!mbar_wait(&ps->land_free[i], ((q / kPrLand) & 1u) ^ 1u, timeout_ns, cta_abort)) {
      pr_fail(ps, cta_abort, fail_where, kWhereEmptyBarrier);
      return false;
    }
    const uint32_t st = land0 + i * kPrLandBytes, st_b = st + (pack_a ? kPrLandPackA : kPrLandA);
    uint64_t* bar = &ps->landed[i];
    mbar_expect_tx(bar, tx);
    const int k0 = kb * kTcBK;
    if (map_a) {
      if (!pack_a) {
        tma_load_2d(st, tmA, k0, row0, bar);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          tma_load_2d(st + (uint32_t)j * (32u * kPrPackA * 4u), tmA, (xa + j * t.k + k0) & ~3, row0 >> 2, bar);
      }
    }
    if (map_b) {
      if (!pack_b) {
        for (int b = 0; b < slabs; ++b)
          tma_load_2d(st_b + (uint32_t)b * kPrSlab, tmB, col0 + 32 * b, k0, bar);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          tma_load_2d(st_b + (uint32_t)j * (8u * kPrPackB * 4u), tmB, (xb + j * n) & ~3, k0 >> 2, bar);
      }
    }
    pend = (pend & ~(3u << (2 * i))) | ((tx ? (1u | (((q / kPrLand) & 1u) << 1)) : 0u) << (2 * i));
  }
  return true;
}

// The producer thread at exit: every copy it issued has landed (bounded,
// whatever the abort flag says), so that none writes the CTA's shared memory
// after it is gone.
__device__ __forceinline__ void pr_produce_quiesce(PrShared* ps, uint32_t pend, uint64_t timeout_ns) {
  volatile uint32_t never = 0;
  for (int i = 0; i < kPrLand; ++i)
    if ((pend >> (2 * i)) & 1u) (void)mbar_wait(&ps->landed[i], (pend >> (2 * i + 1)) & 1u, timeout_ns, &never);
}

// ---------------------------------------------------------------- converters

__device__ __forceinline__ float ld_shared_f32(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
  return v;
}

// Converter warps, landing ql: its operands have landed. Landings also serve
// vector tiles, so that ql runs ahead of the k-step's number q, by an even
// number: both belong to the same group.
__device__ __forceinline__ bool pr_wait_landed(PrShared* ps, uint32_t ql, const uint64_t& timeout_ns, uint32_t* cta_abort,
                                               uint32_t* fail_where) {
  if (mbar_wait_warp<false>(&ps->landed[ql % kPrLand], (ql / kPrLand) & 1u, timeout_ns, cta_abort)) return true;
  if ((threadIdx.x & 31) == 0) pr_fail(ps, cta_abort, fail_where, kWhereEmptyBarrier);
  return false;
}
// Converter warps, k-step q: the MMAs have read its stage's previous k-step, q - 3.
__device__ __forceinline__ bool pr_wait_stage(PrShared* ps, uint32_t q, const uint64_t& timeout_ns, uint32_t* cta_abort,
                                              uint32_t* fail_where) {
  if (!pr_stage_used(q) || mbar_wait_warp<false>(&ps->empty[pr_empty_bar(q - kPrStages)], pr_empty_parity(q - kPrStages),
                                                 timeout_ns, cta_abort))
    return true;
  if ((threadIdx.x & 31) == 0) pr_fail(ps, cta_abort, fail_where, kWhereFullBarrier);
  return false;
}

// Converter warps: split the k-steps of tile t that belong to this warp's
// group (k-step q of the pipeline goes to group q % 2). Warp w of a group takes
// A atoms w + 4 j (8 rows x 32 k) and, of every B slab, k rows 8 w .. +7; a
// lane (r = lane / 4, c = lane % 4) 8 values from column 8 c of row r of each. A
// CTA whose rows all lie beyond A stages only B (its half of the accumulator
// is never stored). Returns false when a wait ran out.
// Both operands aligned:
__device__ __forceinline__ bool pr_convert_aligned(const PrTile t, uint32_t land0, uint32_t st0, PrShared* ps,
                                                   uint32_t it, uint32_t it_l, const uint64_t& timeout_ns,
                                                   uint32_t* cta_abort, uint32_t* fail_where) {
  const int cw = (int)(threadIdx.x >> 5) - kPrConvWarp0, lane = threadIdx.x & 31;
  const int par = cw / kPrGroupWarps, w = cw % kPrGroupWarps;
  const int nkb = (t.k + kTcBK - 1) / kTcBK;
  const int slabs = t.ncols >> 6;
  const bool has_a = t.row0 + (int)ps->cta * 128 < t.m;
  const uint32_t r = (uint32_t)lane >> 2, c = (uint32_t)lane & 3u;
  const uint32_t rd0 = (uint32_t)w * 1024u + r * 128u + (((2u * c) ^ r) << 4);  // and the next chunk at rd0 ^ 16
  const uint32_t wr = swz64(r, c);
  for (int kb = (int)((it + (uint32_t)par) & 1u); kb < nkb; kb += 2) {
    const uint32_t q = it + (uint32_t)kb, ql = it_l + (uint32_t)kb;
    const uint32_t s = pr_stage(q), i = ql % kPrLand;
    if (!pr_wait_landed(ps, ql, timeout_ns, cta_abort, fail_where)) return false;
    const uint32_t ld = land0 + i * kPrLandBytes;
    const uint32_t st = st0 + s * kPrStageBytes;
    // A and the first half of B are read, A is stored, the rest of B is read:
    // 48 values a lane in flight. With all 64 read first the loop spilled.
    uint4 xa[4][2], xb[4][2];
#pragma unroll
    for (int b = 0; b < 4; ++b) xb[b][1].w = 0;
    auto read_b = [&](int b) {
      if (b < slabs) {
        xb[b][0] = ld_shared_v4(ld + kPrLandA + (uint32_t)b * kPrSlab + rd0);
        xb[b][1] = ld_shared_v4(ld + kPrLandA + (uint32_t)b * kPrSlab + (rd0 ^ 16u));
      }
    };
    auto put = [&](const uint4 (&x)[2], uint32_t hi_at, uint32_t lo_at) {
      const float v[8] = {__uint_as_float(x[0].x), __uint_as_float(x[0].y), __uint_as_float(x[0].z),
                          __uint_as_float(x[0].w), __uint_as_float(x[1].x), __uint_as_float(x[1].y),
                          __uint_as_float(x[1].z), __uint_as_float(x[1].w)};
      uint4 hi, lo;
      split8_x2(v, hi, lo);
      st_shared_v4(hi_at, hi);
      st_shared_v4(lo_at, lo);
    };
    if (has_a) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        xa[j][0] = ld_shared_v4(ld + (uint32_t)j * 4096u + rd0);
        xa[j][1] = ld_shared_v4(ld + (uint32_t)j * 4096u + (rd0 ^ 16u));
      }
    }
    read_b(0);
    read_b(1);
    if (!pr_wait_stage(ps, q, timeout_ns, cta_abort, fail_where)) return false;
    if (has_a) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t at = st + (uint32_t)(w + 4 * j) * 512u + wr;
        put(xa[j], at + kPrAOff, at + kPrAlOff);
      }
    }
    read_b(2);
    read_b(3);
    // The landing is free once its values have arrived in registers. An arrive
    // does not wait for loads in flight, a vote on their values does (no lane's
    // value equals both constants, which the compiler does not see).
    const uint32_t last = xb[0][1].w ^ xb[1][1].w ^ xb[2][1].w ^ xb[3][1].w;
    const bool read = (__ballot_sync(0xffffffffu, last == 0x7fa5a5a5u) & __ballot_sync(0xffffffffu, last == 0x7f5a5a5au)) == 0;
    __syncwarp();  // orders the other lanes' reads before lane 0's arrive
    if (lane == 0 && read) mbar_arrive(&ps->land_free[i]);
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      if (b < slabs) {
        const uint32_t at = st + (uint32_t)w * kPrBAtomK + (uint32_t)b * kPrBAtomN + wr;
        put(xb[b], at + kPrBOff, at + kPrBlOff);
      }
    }
    fence_proxy_async_shared();
    __syncwarp();
    if (lane == 0) mbar_arrive_cta(&ps->full[s], 0);
  }
  return true;
}

// Any landing (an operand without a map: every row from global memory), two
// atoms at a time, so that the loop needs no more registers than the aligned
// one.
__device__ __forceinline__ bool pr_convert_packed(const PrTile t, uint32_t land0, uint32_t st0, PrShared* ps, uint32_t it,
                                               uint32_t it_l, const uint64_t& timeout_ns, uint32_t* cta_abort,
                                               uint32_t* fail_where) {
  const int cw = (int)(threadIdx.x >> 5) - kPrConvWarp0, lane = threadIdx.x & 31;
  const int par = cw / kPrGroupWarps, w = cw % kPrGroupWarps;
  const int nkb = (t.k + kTcBK - 1) / kTcBK;
  const int slabs = t.ncols >> 6, m = t.m, k = t.k;
  const int n = (int)t.n;
  const int row0 = t.row0 + (int)ps->cta * 128;
  const int col0 = (int)t.col0 + (int)ps->cta * (t.ncols >> 1);
  const bool has_a = row0 < m;
  const bool map_a = (t.land & kPrMapA) != 0, map_b = (t.land & kPrMapB) != 0;
  const bool pack_a = !map_a || (t.land & kPrPackedA) != 0, pack_b = !map_b || (t.land & kPrPackedB) != 0;
  const float* A = t.A;
  const float* B = t.B;
  const uint32_t r = (uint32_t)lane >> 2, c = (uint32_t)lane & 3u;
  const uint32_t rd0 = (uint32_t)w * 1024u + r * 128u + (((2u * c) ^ r) << 4);
  const uint32_t rd1 = (uint32_t)w * 1024u + r * 128u + (((2u * c + 1u) ^ r) << 4);
  // Packed: row r of an atom is row r % 4 of super-row r / 4 (of the atom's two).
  const uint32_t pj = r & 3u, pi = r >> 2;
  const uint32_t pa = 4u * ((pj * 32u + 2u * (uint32_t)w + pi) * kPrPackA +
                            ((pr_shift(A) + pj * (uint32_t)k) & 3u) + 8u * c);
  const uint32_t pb = 4u * ((pj * 8u + 2u * (uint32_t)w + pi) * kPrPackB +
                            ((pr_shift(B) + pj * (uint32_t)n) & 3u) + 8u * c);
  // Rows of A and k-rows of B in whole super-rows (none without a map).
  const int full_m = map_a ? m & ~3 : 0, full_k = map_b ? k & ~3 : 0;
  const uint32_t wr = swz64(r, c);
  for (int kb = (int)((it + (uint32_t)par) & 1u); kb < nkb; kb += 2) {
    const uint32_t q = it + (uint32_t)kb, ql = it_l + (uint32_t)kb;
    const uint32_t s = pr_stage(q), i = ql % kPrLand;
    if (!pr_wait_landed(ps, ql, timeout_ns, cta_abort, fail_where) ||
        !pr_wait_stage(ps, q, timeout_ns, cta_abort, fail_where))
      return false;
    const uint32_t ld = land0 + i * kPrLandBytes, ld_b = ld + ((t.land & kPrPackedA) ? kPrLandPackA : kPrLandA);
    const uint32_t st = st0 + s * kPrStageBytes;
    auto read = [&](bool packed, uint32_t packed_at, uint32_t a0, uint32_t a1, float (&v)[8]) {
      if (packed) {
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = ld_shared_f32(packed_at + 4u * e);
      } else {
        const uint4 x0 = ld_shared_v4(a0), x1 = ld_shared_v4(a1);
        v[0] = __uint_as_float(x0.x); v[1] = __uint_as_float(x0.y); v[2] = __uint_as_float(x0.z);
        v[3] = __uint_as_float(x0.w); v[4] = __uint_as_float(x1.x); v[5] = __uint_as_float(x1.y);
        v[6] = __uint_as_float(x1.z); v[7] = __uint_as_float(x1.w);
      }
    };
    // 8 values of a row from global memory, zero outside the matrix.
    auto fetch = [](const float* src, bool row_in, int left, float (&v)[8]) {
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = (row_in && e < left) ? __ldcg(src + e) : 0.f;
    };
    float x[2][8];
    if (has_a) {
      const int kk = kb * kTcBK + 8 * (int)c;
#pragma unroll 1
      for (int j0 = 0; j0 < 4; j0 += 2) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const uint32_t j = (uint32_t)(j0 + u);
          read(pack_a, ld + pa + j * (8u * kPrPackA * 4u), ld + j * 4096u + rd0, ld + j * 4096u + rd1, x[u]);
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int j = j0 + u, row = row0 + 8 * (w + 4 * j) + (int)r;
          if (pack_a) {
            if (row >= full_m) {
              fetch(A + (int64_t)row * k + kk, row < m, k - kk, x[u]);
            } else if (kk + 8 > k) {
#pragma unroll
              for (int e = 0; e < 8; ++e)
                if (kk + e >= k) x[u][e] = 0.f;
            }
          }
          const uint32_t at = st + (uint32_t)(w + 4 * j) * 512u + wr;
          uint4 hi, lo;
          split8_x2(x[u], hi, lo);
          st_shared_v4(at + kPrAOff, hi);
          st_shared_v4(at + kPrAlOff, lo);
        }
      }
    }
    const int kr = kb * kTcBK + 8 * w + (int)r;
#pragma unroll 1
    for (int b0 = 0; b0 < slabs; b0 += 2) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const uint32_t b = (uint32_t)min(b0 + u, slabs - 1);
        read(pack_b, ld_b + pb + b * 128u, ld_b + b * kPrSlab + rd0, ld_b + b * kPrSlab + rd1,
             x[u]);
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int b = b0 + u;
        if (b < slabs) {
          if (pack_b && kr >= full_k) {
            const int col = col0 + 32 * b + 8 * (int)c;
            fetch(B + (int64_t)kr * n + col, kr < k, n - col, x[u]);
          }
          const uint32_t at = st + (uint32_t)w * kPrBAtomK + (uint32_t)b * kPrBAtomN + wr;
          uint4 hi, lo;
          split8_x2(x[u], hi, lo);
          st_shared_v4(at + kPrBOff, hi);
          st_shared_v4(at + kPrBlOff, lo);
        }
      }
    }
    fence_proxy_async_shared();
    __syncwarp();
    if (lane == 0) {
      mbar_arrive(&ps->land_free[i]);
      mbar_arrive_cta(&ps->full[s], 0);
    }
  }
  return true;
}

__device__ __forceinline__ bool pr_convert(const PrTile t, uint8_t* land, uint8_t* stages, PrShared* ps, uint32_t it,
                                           uint32_t it_l, const uint64_t& timeout_ns, uint32_t* cta_abort,
                                           uint32_t* fail_where) {
  const uint32_t land0 = smem_u32(land), st0 = smem_u32(stages);
  if (t.land == (kPrMapA | kPrMapB))
    return pr_convert_aligned(t, land0, st0, ps, it, it_l, timeout_ns, cta_abort, fail_where);
  return pr_convert_packed(t, land0, st0, ps, it, it_l, timeout_ns, cta_abort, fail_where);
}

// ---------------------------------------------------------------- vector tiles
//
// A CTA's part of a vector-add or vector-multiply tile runs through the landing
// ring as well: the producer lands 4096 elements of a and of b at a time (two
// bulk copies of 16 KB), the converter group of the landing adds or multiplies
// them and stores c. The copies of a tile are under way while the tile before
// is worked on, 128 KB a CTA. With direct loads (16-byte loads, four of each
// operand a thread in flight, drained at every tile's end) 16 x 4 vector adds
// of 2^22 took 0.66 ms a launch on CTA pairs.

constexpr int kPrVecChunk = 4096;  // elements per landing
constexpr uint32_t kPrVecB = kPrVecChunk * 4;
static_assert(2 * kPrVecB <= kPrLandBytes, "a vector chunk fits a landing");

// Landings of `len` elements: an even number, so that landings and stages of
// the same index parity stay with the same converter group.
__device__ __forceinline__ uint32_t pr_vec_chunks(int64_t len) {
  return ((uint32_t)((len + kPrVecChunk - 1) / kPrVecChunk) + 1u) & ~1u;
}

// Copy of `bytes` (a multiple of 16) from global to this CTA's shared memory,
// counted on `bar`; both addresses 16-byte aligned.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// The producer thread: land a[0 .. len-1] and b[0 .. len-1] (16-byte aligned)
// but for the last len % 4 elements.
__device__ __forceinline__ bool pr_vec_produce(const float* a, const float* b, int64_t len, uint8_t* land, PrShared* ps,
                                               uint32_t it_l, uint64_t timeout_ns, uint32_t* cta_abort,
                                               uint32_t* fail_where, uint32_t& pend) {
  const uint32_t n = pr_vec_chunks(len), land0 = smem_u32(land);
  for (uint32_t ch = 0; ch < n; ++ch) {
    const uint32_t q = it_l + ch, i = q % kPrLand;
    if (!mbar_wait(&ps->land_free[i], ((q / kPrLand) & 1u) ^ 1u, timeout_ns, cta_abort)) {
      pr_fail(ps, cta_abort, fail_where, kWhereEmptyBarrier);
      return false;
    }
    const int64_t at = (int64_t)ch * kPrVecChunk;
    const int64_t left = len - at;
    const uint32_t bytes = left >= kPrVecChunk ? kPrVecB : left > 0 ? (uint32_t)(left >> 2) * 16u : 0u;
    uint64_t* bar = &ps->landed[i];
    mbar_expect_tx(bar, 2 * bytes);
    if (bytes) {
      const uint32_t st = land0 + i * kPrLandBytes;
      bulk_g2s(st, a + at, bytes, bar);
      bulk_g2s(st + kPrVecB, b + at, bytes, bar);
    }
    pend = (pend & ~(3u << (2 * i))) | ((bytes ? (1u | (((q / kPrLand) & 1u) << 1)) : 0u) << (2 * i));
  }
  return true;
}

// Converter warps: c = a op b over the landings of this warp's group; whole
// landings run unrolled (64 vector multiplies of 2^22 593 to 540 us a launch).
template <int OP>
__device__ __forceinline__ bool pr_vec_convert(const float* a, const float* b, float* c, int64_t len, int iters,
                                               uint8_t* land, PrShared* ps, uint32_t it_l, uint64_t timeout_ns,
                                               uint32_t* cta_abort, uint32_t* fail_where) {
  const int cw = (int)(threadIdx.x >> 5) - kPrConvWarp0, lane = threadIdx.x & 31;
  const uint32_t par = (uint32_t)(cw / kPrGroupWarps), t = (uint32_t)(cw % kPrGroupWarps) * 32 + lane;
  const uint32_t n = pr_vec_chunks(len), land0 = smem_u32(land);
  const bool cvec = (reinterpret_cast<uintptr_t>(c) & 15) == 0;
  for (uint32_t ch = (it_l + par) & 1u; ch < n; ch += 2) {
    const uint32_t q = it_l + ch;
    if (!mbar_wait_warp<false>(&ps->landed[q % kPrLand], (q / kPrLand) & 1u, timeout_ns, cta_abort)) {
      if (lane == 0) pr_fail(ps, cta_abort, fail_where, kWhereEmptyBarrier);
      return false;
    }
    const int64_t at = (int64_t)ch * kPrVecChunk, left = len - at;
    const uint32_t n4 = left >= kPrVecChunk ? kPrVecChunk / 4 : left > 0 ? (uint32_t)(left >> 2) : 0u;
    const uint32_t st = land0 + (q % kPrLand) * kPrLandBytes + 16u * t;
    auto four = [&](uint32_t j) {  // the thread's j-th four elements
      const uint4 xu = ld_shared_v4(st + j * (16u * 32 * kPrGroupWarps));
      const uint4 yu = ld_shared_v4(st + kPrVecB + j * (16u * 32 * kPrGroupWarps));
      return elem_op4<OP>(*reinterpret_cast<const float4*>(&xu), *reinterpret_cast<const float4*>(&yu), iters);
    };
    float* dst = c + at + 4 * (int64_t)t;
    constexpr uint32_t kAll = kPrVecChunk / (4 * 32 * kPrGroupWarps);
    if (cvec && left >= kPrVecChunk) {
#pragma unroll 8
      for (uint32_t j = 0; j < kAll; ++j) __stcs(reinterpret_cast<float4*>(dst + j * (4 * 32 * kPrGroupWarps)), four(j));
    } else {
#pragma unroll 1
      for (uint32_t j = 0; t + j * (32 * kPrGroupWarps) < n4; ++j) {
        const float4 z = four(j);
        float* d = dst + j * (4 * 32 * kPrGroupWarps);
        if (cvec) {
          __stcs(reinterpret_cast<float4*>(d), z);
        } else {
          d[0] = z.x;
          d[1] = z.y;
          d[2] = z.z;
          d[3] = z.w;
        }
      }
    }
    if (left > 0 && left < kPrVecChunk) {  // the last elements, not landed
      const int64_t e = at + 4 * (int64_t)n4 + t;
      if (e < len) c[e] = elem_op<OP>(__ldcg(a + e), __ldcg(b + e), iters);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&ps->land_free[q % kPrLand]);
  }
  return true;
}

// ---------------------------------------------------------------- MMA

// Leader, the MMA thread: tile t into accumulator (tile_no & 1)
// once the epilogues of both CTAs have drained it. *wait_acc (may be NULL)
// sums the SM clocks waited for staged k-steps. Returns false when a wait ran
// out.
__device__ __forceinline__ bool pr_mma(const PrTile t, uint8_t* stages, PrShared* ps, uint32_t it, uint32_t tile_no,
                                       uint64_t timeout_ns, uint32_t* cta_abort, uint32_t* fail_where,
                                       uint64_t* wait_acc) {
  const uint32_t b = tile_no & 1u;
  if (!mbar_wait(&ps->acc_empty[b], ((tile_no >> 1) & 1u) ^ 1u, timeout_ns, cta_abort)) {
    pr_fail(ps, cta_abort, fail_where, kWhereAccumBarrier);
    return false;
  }
  tc_fence_after();
  const uint32_t tmem = ps->tmem_base + b * (uint32_t)kPrN;
  const uint32_t idesc = idesc_bf16_f32(kPrM, 0) | (1u << 16) | ((uint32_t)(t.ncols >> 3) << 17);
  const int nkb = (t.k + kTcBK - 1) / kTcBK;
  const uint32_t st0 = smem_u32(stages);
  for (int kb = 0; kb < nkb; ++kb) {
    const uint32_t q = it + (uint32_t)kb, s = pr_stage(q), ph = pr_full_parity(q);
    const long long c0 = wait_acc != nullptr ? clock64() : 0;
    if (!mbar_wait(&ps->full[s], ph, timeout_ns, cta_abort)) {
      pr_fail(ps, cta_abort, fail_where, kWhereFullBarrier);
      return false;
    }
    if (wait_acc != nullptr) *wait_acc += (uint64_t)(clock64() - c0);
    tc_fence_after();
    const uint32_t sb = st0 + s * kPrStageBytes;
    const uint64_t dAh = sdesc_k64b(sb + kPrAOff), dAl = sdesc_k64b(sb + kPrAlOff);
    const uint64_t dBh = pr_desc_b(sb + kPrBOff), dBl = pr_desc_b(sb + kPrBlOff);
#pragma unroll
    for (int kk = 0; kk < kTcBK / 16; ++kk) {
      const uint64_t adv_a = (uint64_t)(kk * 32) >> 4;             // 16 bf16 = 32 bytes along a K-major row
      const uint64_t adv_b = (uint64_t)(kk * 2 * kPrBAtomK) >> 4;  // two 8-row k groups of B
      umma_bf16_pair(tmem, dAl + adv_a, dBh + adv_b, idesc, (kb | kk) ? 1u : 0u);
      umma_bf16_pair(tmem, dAh + adv_a, dBl + adv_b, idesc, 1u);
      umma_bf16_pair(tmem, dAh + adv_a, dBh + adv_b, idesc, 1u);
    }
    umma_commit_pair(&ps->empty[pr_empty_bar(q)]);
  }
  umma_commit_pair(&ps->acc_full[b]);
  return true;
}

// ---------------------------------------------------------------- epilogue

// 32 x 32 transpose across a warp: on entry lane l holds row l in r[0..31],
// on return lane l holds column l (r[i] = element l of row i).
__device__ __forceinline__ void warp_transpose32(uint32_t (&r)[32], int lane) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    const bool up = (lane & d) != 0;
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      if (i & d) continue;
      const uint32_t send = up ? r[i] : r[i + d];
      const uint32_t got = __shfl_xor_sync(0xffffffffu, send, d);
      if (up) r[i] = got;
      else r[i + d] = got;
    }
  }
}

// Epilogue warps: this CTA's 128 rows of accumulator (tile_no & 1) into C,
// 32 columns at a time; TMEM hands each thread a row, stored as whole 32-byte
// sectors (16-byte stores when n is a multiple of 4 only). With other row
// lengths rows start anywhere: a block is transposed across the warp so that
// each store writes 32 consecutive values of a row. Then frees the
// accumulator. Returns the %globaltimer when the accumulator was complete, 0
// when the wait for it ran out.
__device__ __forceinline__ uint64_t pr_epilogue(const PrTile t, PrShared* ps, uint32_t tile_no, uint64_t timeout_ns,
                                                uint32_t* cta_abort, uint32_t* fail_where) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t b = tile_no & 1u;
  if (!mbar_wait_warp<false>(&ps->acc_full[b], (tile_no >> 1) & 1u, timeout_ns, cta_abort)) {
    if (lane == 0) pr_fail(ps, cta_abort, fail_where, kWhereAccumBarrier);
    return 0;
  }
  const uint64_t t0 = globaltimer();
  tc_fence_after();
  const int wrow = t.row0 + (int)ps->cta * 128 + 32 * w;  // the warp's first row
  const int row = wrow + lane;
  const uintptr_t ca = reinterpret_cast<uintptr_t>(t.C);
  const int vec = ((t.n & 7) == 0 && (ca & 31) == 0) ? 2 : ((t.n & 3) == 0 && (ca & 15) == 0) ? 1 : 0;
  const uint32_t taddr = ps->tmem_base + b * (uint32_t)kPrN + ((uint32_t)(w * 32) << 16);
  const int chunks = wrow < t.m ? t.ncols >> 5 : 0;
  auto store_chunk = [&](int ch, uint32_t (&r)[32]) {
    const int64_t c0 = t.col0 + ch * 32;
    if (c0 >= t.n) return;
    if (vec != 0 && c0 + 32 <= t.n) {
      if (row < t.m) {
        float* dst = t.C + (int64_t)row * t.n + c0;
        if (vec == 2) {
#pragma unroll
          for (int j = 0; j < 4; ++j) st_v8(dst + 8 * j, r + 8 * j);
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j)
            reinterpret_cast<uint4*>(dst)[j] = make_uint4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
        }
      }
    } else {
      warp_transpose32(r, lane);
      const int rows = min(32, t.m - wrow);
      float* dst = t.C + (int64_t)wrow * t.n + c0 + lane;
      if (c0 + lane < t.n) {
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (i < rows) dst[(int64_t)i * t.n] = __uint_as_float(r[i]);
      }
    }
  };
#pragma unroll 1
  for (int ch = 0; ch < chunks; ch += 2) {  // chunks is even
    uint32_t r0[32], r1[32];
    __syncwarp();
    tmem_ld_32x32b_x32(taddr + (uint32_t)(ch * 32), r0);
    tmem_ld_32x32b_x32(taddr + (uint32_t)((ch + 1) * 32), r1);
    tmem_ld_wait();
    store_chunk(ch, r0);
    store_chunk(ch + 1, r1);
  }
  tc_fence_before();
  __syncwarp();
  if (lane == 0) mbar_arrive_cta(&ps->acc_empty[b], 0);
  return t0;
}

}  // namespace gvm
