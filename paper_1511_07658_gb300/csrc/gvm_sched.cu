// Persistent scheduler of the GPU virtualization manager.
//
// The paper's manager (Section 5) is a daemon that owns the only GPU context,
// takes requests from per-process queues, waits at a request barrier and
// flushes every process's stream so that kernels and copies of different
// processes overlap (Section 4.2.2). Here the request queues are rings of task
// descriptors in pinned host memory, one per rank, and the manager's request
// loop is this kernel: its CTAs take descriptors from the rings (round robin
// over ranks, FIFO within a rank), cut each task into tiles, and run tiles of
// all ranks' tasks side by side -- the concurrency the paper gets from one
// stream per process, without a kernel launch per task.
//
// Work flow per CTA:
//   claim:   every queue entry covers a contiguous range of one global tile
//            space; a CTA takes the next tile index with one atomicAdd on
//            next_tile and finds its entry by a short forward search. An
//            index beyond the published tiles is a reservation the CTA waits
//            for (ingesting meanwhile). Warp 0 claims the next tile while the
//            other warps run the current one.
//   ingest:  one CTA at a time (holding a lock) copies ready descriptors from
//            the host rings into the device task table and appends queue
//            entries.
//   finish:  the CTA that completes a task's last tile publishes completion:
//            the host completion word (resident tasks) or the device done word
//            on which the rank's output-copy stream waits (host-buffer tasks).
//
// Every wait is bounded (wait_timeout_ns); a wait that runs out records a
// status word in host memory and stops the kernel. In continuous mode the
// kernel stays resident until the host sets the stop word (idle CTAs sleep
// idle_poll_ns between polls); in barrier (drain) mode it exits once every
// descriptor published before its launch has been taken.
#include "gvm_device.cuh"
#include <cstddef>

#include "gvm_pair.cuh"
#include "gvm_runtime.h"

namespace gvm {

constexpr uint32_t kMaxQuantum = 8;

// FMA path: two tile slots; the CTA runs the tile in one while warp 0 claims
// the next into the other. go: 1 = a tile is there, 0 = exit, 2 = nothing
// claimed yet.
struct alignas(128) SchedShared {
  TaskBody body[2];  // copies of the claimed tasks' bodies
  uint32_t go[2];
  uint32_t task[2];
  uint32_t tile[2];
  uint64_t t_tile;   // when the current tile began (thread 0)
  uint64_t prof[kProfSlots];  // this CTA's phase counters (kProf*), written by thread 0 only
  uint64_t claim[4];  // Claim state (see acquire), owned by warp 0
  uint32_t list[32 * kMaxQuantum];  // ingest's scratch, warp 0
};

constexpr uint64_t kLookaheadTiles = 512;  // ingest ahead when this few published tiles remain
constexpr uint64_t kQuietNs = 20000; // skip look-ahead ingest this long after an empty pass

__device__ __forceinline__ uint32_t ld_volatile_u32(const uint32_t* p) {
  return *reinterpret_cast<const volatile uint32_t*>(p);
}

__device__ void report_error(const SchedParams& p, uint32_t status, uint32_t where, uint32_t info) {
  HostShared* hs = p.host_shared;
  *reinterpret_cast<volatile uint32_t*>(&hs->where) = where;
  *reinterpret_cast<volatile uint32_t*>(&hs->info) = info;
  __threadfence_system();
  st_release_sys(&hs->status, status);
  atomicExch(&p.ctrl->abort, 1u);
}

// Marks task idx complete: timestamps, then the word its waiter watches.
__device__ void complete_task(const SchedParams& p, uint32_t idx, uint32_t tag, uint32_t flags,
                              uint64_t t_ingest) {
  HostComplete* hc = &p.host_complete[idx];
  const uint64_t now = globaltimer();
  st_relaxed_sys64(&hc->t_ingest, t_ingest);
  st_relaxed_sys64(&hc->t_done, now);
  atomicMax(reinterpret_cast<unsigned long long*>(&p.ctrl->t_last_done), (unsigned long long)now);
  if (flags & kFlagNeedsD2H) {  // releases: all of the above, and the task's results, before the word
    st_release_sys(&p.done[idx], tag);
  } else {
    st_release_sys(&hc->tag, tag);
  }
}

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += o;
  }
  return v;
}

struct IngestOut {
  uint32_t locked_out;
  uint32_t published;
  uint32_t pending;
};

// The task fields are a descriptor's last 128 bytes, the tensor maps its
// first 256.
constexpr uint32_t kFieldsAt = 256;
static_assert(offsetof(TaskBody, type) == kFieldsAt && sizeof(TaskBody) == 384, "TaskBody fields");
static_assert(offsetof(TaskBody, flags) == 260 && offsetof(TaskBody, tag) == 272 && offsetof(TaskBody, ntiles) == 276,
              "TaskBody header words");
static_assert(offsetof(TaskBody, tmA) == 0 && offsetof(TaskBody, tmB) == 128 && sizeof(CUtensorMap) == 128,
              "TaskBody maps");

// Check word of a queue entry: a reader may meet an entry that is being
// written (one beyond the published tiles) and must not take a mixture of
// its old and new words for a whole entry.
__device__ __forceinline__ uint32_t pub_check(uint32_t base, uint32_t seq, uint32_t task, uint32_t cnt) {
  return base ^ (seq * 0x9e3779b9u) ^ (task << 16) ^ cnt;
}

// One warp copies the descriptors of n tasks from the host ring to the device
// table: the fields (8 pieces of 16 bytes) of all, the maps (16 pieces) of those
// marked kListMaps; kBatch reads of host memory in flight a lane (a round trip
// takes 3 us).
constexpr uint32_t kListMaps = 1u << 31;
template <uint32_t kBatch>
__device__ __forceinline__ void copy_bodies(const SchedParams& p, const uint32_t* list, uint32_t n, bool any_maps) {
  const uint32_t lane = threadIdx.x & 31, split = n * 8, total = split + (any_maps ? n * 16 : 0);
  // Piece u: the task, and its place in the descriptor; false: nothing to copy.
  auto place = [&](uint32_t u, uint32_t& idx, uint32_t& at) -> bool {
    if (u >= total) return false;
    const uint32_t w = u - split;
    const uint32_t e = u < split ? list[u / 8] : list[w / 16];
    idx = e & ~kListMaps;
    at = u < split ? kFieldsAt + 16 * (u % 8) : 16 * (w % 16);
    return u < split || (e & kListMaps);
  };
#pragma unroll 1
  for (uint32_t u0 = lane; u0 < total; u0 += 32 * kBatch) {
    uint4 v[kBatch];
    uint32_t idx, at;
#pragma unroll
    for (uint32_t j = 0; j < kBatch; ++j)
      if (place(u0 + 32 * j, idx, at)) v[j] = ld_volatile_v4(reinterpret_cast<const uint8_t*>(&p.host_desc[idx]) + at);
#pragma unroll
    for (uint32_t j = 0; j < kBatch; ++j)
      if (place(u0 + 32 * j, idx, at)) st_cg_v4(reinterpret_cast<uint8_t*>(&p.tasks[idx].body) + at, v[j]);
  }
}

// Warp 0 of one CTA: move ready descriptors from the host rings into the
// device table and append their queue entries, each covering a contiguous
// range of the global tile space. All lanes call. Lane = rank: it reads the
// heads and the header words of its rank's next tasks (kBatch tasks' reads in
// flight), then the warp copies all taken descriptors together. Read and
// stored task by task by each lane, a pass of 64 tasks with tensor maps took
// 43 us, 0.68 ms of a 1024-task launch. list: 32 x kMaxQuantum words in shared
// memory.
template <uint32_t kBatch>
__device__ __forceinline__ IngestOut ingest_pass(const SchedParams& p, uint64_t* prof, uint32_t* list) {
  const int lane = threadIdx.x & 31;
  IngestOut out{0, 0, 0};
  uint32_t got = 0;
  if (lane == 0) got = (atomicCAS(&p.ctrl->ingest_lock, 0u, 1u) == 0u) ? 1u : 0u;
  got = __shfl_sync(0xffffffffu, got, 0);
  if (!got) {
    out.locked_out = 1;
    return out;
  }
  __threadfence();
  // Drain mode: once a pass has found the rings empty (`drained`, set below
  // under this lock), nothing more is published in this launch, even if the
  // host has published descriptors since: CTAs leave with reservations
  // beyond the published tiles, and a tile published after its reserver
  // left would never run. Those descriptors wait in the rings for the next
  // launch.
  const uint32_t closed = ld_relaxed_gpu(&p.ctrl->drained);
  const uint64_t pub0 = ld_relaxed_gpu64(&p.ctrl->published);
  const uint64_t tiles0 = ld_relaxed_gpu64(&p.ctrl->published_tiles);
  const uint64_t consumed = ld_relaxed_gpu64(&p.ctrl->cursor);
  const uint32_t rr = ld_relaxed_gpu(&p.ctrl->rr);
  if (p.drain && __shfl_sync(0xffffffffu, closed, 0)) {
    if (lane == 0) {
      __threadfence();
      atomicExch(&p.ctrl->ingest_lock, 0u);
    }
    __syncwarp();
    return out;
  }
  const uint64_t now = globaltimer();
  uint64_t pub = pub0, ptiles = tiles0;
  uint32_t pending = 0;
  bool bad = false;

  for (uint32_t g = 0; g < p.ranks; g += 32) {
    // Keep at most half the ring between the hand-out frontier and the
    // newest entry, so that an entry is read long before its slot is reused.
    const uint64_t used = pub - consumed;
    const uint32_t space = used < p.qcap / 2 ? (uint32_t)(p.qcap / 2 - used) : 0u;
    uint32_t quantum = min(p.quantum, kMaxQuantum);
    const uint32_t lanes = min(32u, p.ranks - g);
    if (lanes * quantum > space) quantum = space / lanes;

    uint32_t r = 0, t = 0, take = 0, avail = 0, lim = 0;
    uint32_t tcnt[kMaxQuantum];  // tiles of the taken tasks (0: nothing to publish); indexed statically
    uint32_t entries = 0, tiles = 0, maps = 0;  // maps: bit i = task i has tensor maps to copy
    const bool valid = (g + lane) < p.ranks;
    if (valid) {
      r = (rr + g + lane) % p.ranks;
      const uint32_t h = ld_acquire_sys(&p.host_heads[r].head);
      t = ld_relaxed_gpu(&p.tail[r]);
      avail = h - t;
      lim = min(avail, quantum);
    }
    bool more = valid;
#pragma unroll
    for (uint32_t base = 0; base < kMaxQuantum; base += kBatch) {
      if (!__any_sync(0xffffffffu, more && base < lim)) {
#pragma unroll
        for (uint32_t i = 0; i < kBatch; ++i) tcnt[base + i] = 0;
        continue;
      }
      uint4 h0[kBatch], h1[kBatch];
      uint32_t rdy[kBatch];
#pragma unroll
      for (uint32_t i = 0; i < kBatch; ++i) {
        if (more && base + i < lim) {
          const uint32_t idx = r * p.depth + ((t + base + i) & (p.depth - 1));
          const uint4* src = reinterpret_cast<const uint4*>(&p.host_desc[idx]) + kFieldsAt / 16;
          h0[i] = ld_volatile_v4(src);      // type, flags, rank, slot
          h1[i] = ld_volatile_v4(src + 1);  // tag, ntiles
          rdy[i] = ld_relaxed_gpu(&p.ready[idx]);
        }
      }
#pragma unroll
      for (uint32_t i = 0; i < kBatch; ++i) {
        tcnt[base + i] = 0;
        if (more && base + i < lim) {
          const uint32_t s = t + base + i;
          const uint32_t idx = r * p.depth + (s & (p.depth - 1));
          const uint32_t flags = h0[i].y, tag = h1[i].x, ntiles = h1[i].y;
          if ((flags & kFlagNeedsReady) && rdy[i] != s + 1u) {
            more = false;
          } else {
            ++take;
            if (tag != s + 1u) {
              bad = true;
            } else {
              DevTask* dt = &p.tasks[idx];
              *reinterpret_cast<volatile uint32_t*>(&dt->tiles_done) = 0;
              *reinterpret_cast<volatile uint64_t*>(&dt->t_ingest) = now;
              if (ntiles == 0) {
                __threadfence();
                complete_task(p, idx, tag, flags, now);
              } else {
                if (flags & (kFlagTmA | kFlagTmB)) maps |= 1u << (base + i);
                tcnt[base + i] = ntiles;
                ++entries;
                tiles += ntiles;
              }
            }
          }
        }
      }
    }
    // The ready words (written by the input streams after their copies) were
    // read relaxed: order the copies' data before what is published below.
    __threadfence();

    // Queue entries, and the list of what to copy.
    const uint32_t ie = warp_incl_scan(entries), it = warp_incl_scan(tiles);
    const uint32_t te = __shfl_sync(0xffffffffu, ie, 31), tt = __shfl_sync(0xffffffffu, it, 31);
    uint64_t e0 = pub + ie - entries, b0 = ptiles + it - tiles;
    uint32_t at = ie - entries;
#pragma unroll
    for (uint32_t i = 0; i < kMaxQuantum; ++i) {
      if (!tcnt[i]) continue;
      const uint32_t idx = r * p.depth + ((t + i) & (p.depth - 1));
      list[at++] = idx | (((maps >> i) & 1u) ? kListMaps : 0u);
      uint4* pe = reinterpret_cast<uint4*>(&p.pubq[e0 & (p.qcap - 1)]);
      st_cg_v4(pe, make_uint4((uint32_t)b0, (uint32_t)(b0 >> 32), (uint32_t)e0, (uint32_t)(e0 >> 32)));
      st_cg_v4(pe + 1, make_uint4(idx, 0, tcnt[i], pub_check((uint32_t)b0, (uint32_t)e0, idx, tcnt[i])));
      ++e0;
      b0 += tcnt[i];
    }
    __syncwarp();
    copy_bodies<2 * kBatch>(p, list, te, __any_sync(0xffffffffu, maps != 0));
    __syncwarp();
    if (valid && take > 0) *reinterpret_cast<volatile uint32_t*>(&p.tail[r]) = t + take;
    pending += avail - take;
    pub += te;
    ptiles += tt;
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) pending += __shfl_xor_sync(0xffffffffu, pending, d);
  const uint32_t any_bad = __any_sync(0xffffffffu, bad);
  __threadfence();
  fence_tensormap_release();
  __syncwarp();
  if (lane == 0) {
    if (pending == 0 && pub == pub0) {
      *reinterpret_cast<volatile uint64_t*>(&p.ctrl->quiet_until) = now + kQuietNs;
      if (p.drain) st_release_gpu(&p.ctrl->drained, 1u);  // under the lock: no later pass publishes
    }
    *reinterpret_cast<volatile uint32_t*>(&p.ctrl->rr) = (rr + 1) % p.ranks;
    if (pub != pub0) {
      *reinterpret_cast<volatile uint64_t*>(&p.ctrl->published) = pub;
      st_release_gpu64(&p.ctrl->published_tiles, ptiles);
    }
    st_release_gpu(&p.ctrl->ingest_lock, 0u);
    if (any_bad) report_error(p, kStatusBadTask, 0, 0);
  }
  __syncwarp();
  out.published = (uint32_t)(pub - pub0);
  out.pending = pending;
  if (lane == 0 && out.published) {
    prof[kProfIngest] += globaltimer() - now;
    prof[kProfIngests] += 1;
  }
  return out;
}

// The pair scheduler calls it (kCall): inlined twice into its claim loop, its
// registers spilled there, and what spills is read back from L2 (the claim's
// own acquires invalidate L1). In the FMA scheduler a call would cost the tile
// loop its registers.
static __device__ __noinline__ IngestOut ingest_call(const SchedParams& p, uint64_t* prof, uint32_t* list) {
  return ingest_pass<4>(p, prof, list);
}
template <bool kCall>
__device__ __forceinline__ IngestOut ingest(const SchedParams& p, uint64_t* prof, uint32_t* list) {
  if constexpr (kCall) return ingest_call(p, prof, list);
  else return ingest_pass<1>(p, prof, list);
}

__device__ __forceinline__ uint32_t bcast(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }
__device__ __forceinline__ uint64_t bcast64(uint64_t v) {
  const uint32_t lo = __shfl_sync(0xffffffffu, (uint32_t)v, 0);
  const uint32_t hi = __shfl_sync(0xffffffffu, (uint32_t)(v >> 32), 0);
  return ((uint64_t)hi << 32) | lo;
}

// A CTA's claim state, kept in shared memory across calls: a tile index
// handed out by next_tile that may lie beyond the published tiles (then the
// CTA waits for it, ingesting meanwhile), and where its entry search resumes.
struct Claim {
  uint64_t resv;     // reserved tile index
  uint64_t hint;     // queue entry to start the next search at
  uint64_t stall_since;  // when published descriptors started waiting for their inputs (0: not waiting)
  uint32_t has_resv;
  uint32_t pad;
};

// One warp: find the next tile to run. Returns 1 with (task, tile) set,
// 0 when the kernel should exit, and 2 when the reserved tile is not
// published yet and either !blocking or a blocking call has found nothing for
// idle_return_ns (0: never). Decisions use values that one lane read and
// broadcast, so the warp never diverges across the shuffles.
//
// Claiming is one atomicAdd on next_tile per tile: there is no per-entry
// counter for all CTAs to contend on. A tile beyond published_tiles is a
// reservation; tiles are published in increasing order, so it becomes valid
// without further claims.
//
// The control words are read by different lanes at once, an entry window in
// one go: a claim is three round trips to L2 with the task's fields (read by
// the caller). Read one after another they were about ten: a claim took 10 us
// of a loaded GPU, longer than a 256 x 256 x 512 tile.
template <bool kCall>
__device__ __forceinline__ int acquire(const SchedParams& p, Claim* cl, uint32_t* list, uint32_t& task, uint32_t& tile,
                                       uint64_t* prof, bool blocking, uint64_t idle_return_ns = 0) {
  const int lane = threadIdx.x & 31;
  uint64_t entered = 0;
  auto set_stall = [&](uint64_t v) {
    if (lane == 0) cl->stall_since = v;
    __syncwarp();
  };
  while (true) {
    uint64_t v = 0;
    if (lane == 0) {
      if (!cl->has_resv) {
        cl->resv = atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->next_tile), 1ull);
        cl->has_resv = 1;
      }
      v = cl->resv;
    } else if (lane == 1) {
      v = ld_relaxed_gpu(&p.ctrl->abort);
    } else if (lane == 2) {
      v = ld_acquire_gpu(&p.ctrl->drained);
    } else if (lane == 3) {
      v = ld_acquire_gpu64(&p.ctrl->published_tiles);
    } else if (lane == 4) {
      v = ld_relaxed_gpu64(&p.ctrl->quiet_until);
    } else if (lane == 5) {
      v = globaltimer();
    }
    __syncwarp();
    const uint64_t x = __shfl_sync(0xffffffffu, v, 0), pt = __shfl_sync(0xffffffffu, v, 3);
    const uint64_t quiet = __shfl_sync(0xffffffffu, v, 4), now = __shfl_sync(0xffffffffu, v, 5);
    if (__shfl_sync(0xffffffffu, v, 1)) return 0;
    const bool drained = __shfl_sync(0xffffffffu, v, 2) != 0;
    if (entered == 0) entered = now;
    const bool here = x < pt;
    // The reserved tile is not published yet. Before leaving, look at the
    // published tiles once more: another CTA's last ingest pass may have
    // published the reserved tile since pt was read, and a tile whose owner
    // leaves would never run. Once the rings are drained (or stop is set with
    // nothing pending) no further tile is published, so this read is final.
    auto reserved_published = [&]() -> bool {
      uint64_t pt2 = 0;
      if (lane == 0) pt2 = ld_acquire_gpu64(&p.ctrl->published_tiles);
      return x < bcast64(pt2);
    };
    if (!here && p.drain && drained) {
      if (reserved_published()) continue;
      return 0;
    }
    // Ingest when the tile is not there, or to keep the queue ahead of the CTAs.
    IngestOut r{0, 0, 0};
    if (!here || (pt - x <= kLookaheadTiles && now >= quiet)) r = ingest<kCall>(p, prof, list);
    if (here) {
      // Find the entry holding tile x: the last entry with base <= x. Entries
      // are published in tile order, and x only grows from one claim of a CTA
      // to the next, so the search starts at the entry of this CTA's previous
      // tile; the warp checks 32 entries per step. An ingest pass releases
      // published_tiles only after writing its entries, so those up to the one
      // holding x are whole; a later one may be half written, which its check
      // word shows, or whole, with a base above x.
      uint32_t etask = 0, off = 0, ok = 1;
      uint64_t e0 = 0;
      if (lane == 0) e0 = cl->hint;
      e0 = bcast64(e0);
      while (true) {
        const uint64_t e = e0 + (uint64_t)lane;
        const PubEntry* pe = &p.pubq[e & (p.qcap - 1)];
        const uint4 w0 = ld_volatile_v4(pe), w1 = ld_volatile_v4(reinterpret_cast<const uint4*>(pe) + 1);
        const uint64_t base = ((uint64_t)w0.y << 32) | w0.x, seq = ((uint64_t)w0.w << 32) | w0.z;
        const bool le = (seq == e) && base <= x && w1.w == pub_check(w0.x, w0.z, w1.x, w1.z);
        const uint32_t m = __ballot_sync(0xffffffffu, le);
        if (m == 0) {  // not even the first entry starts at or before x
          ok = 0;
          break;
        }
        const int last = 31 - __clz(m);
        if (last == 31 && (m & 1u)) {  // the whole window precedes x: move on
          e0 += 31;
          continue;
        }
        const uint64_t hit_base = __shfl_sync(0xffffffffu, base, last);
        const uint32_t hit_cnt = __shfl_sync(0xffffffffu, w1.z, last);
        etask = __shfl_sync(0xffffffffu, w1.x, last);
        if (x >= hit_base + hit_cnt) {  // a hole in the tile space: the ring bound was broken
          ok = 0;
          break;
        }
        off = (uint32_t)(x - hit_base);
        if (lane == 0) {
          const uint64_t ehit = e0 + (uint64_t)last;
          if (x + 1 == hit_base + hit_cnt)
            atomicMax(reinterpret_cast<unsigned long long*>(&p.ctrl->cursor), (unsigned long long)(ehit + 1));
          cl->hint = ehit;
          cl->has_resv = 0;
          cl->stall_since = 0;
        }
        __syncwarp();
        break;
      }
      if (!ok) {
        if (lane == 0) report_error(p, kStatusBadTask, kWhereQueueFull, (uint32_t)x);
        __syncwarp();
        return 0;
      }
      task = etask;
      tile = off;
      return 1;
    }
    if (r.published) {
      set_stall(0);
      continue;
    }
    if (!r.locked_out) {
      if (r.pending == 0) {
        set_stall(0);
        if (p.drain) {  // this pass (or an earlier one) closed the launch: `drained` is set
          if (reserved_published()) continue;
          return 0;
        }
        uint32_t stop = 0;
        if (lane == 0) stop = ld_acquire_sys(&p.host_shared->stop);
        if (bcast(stop)) {
          if (reserved_published()) continue;
          return 0;
        }
      } else if (blocking) {
        uint64_t since = 0;
        if (lane == 0) {
          if (cl->stall_since == 0) cl->stall_since = now;
          since = cl->stall_since;
        }
        since = bcast64(since);
        if (now - since > p.wait_timeout_ns) {
          if (lane == 0) report_error(p, kStatusTimeout, kWhereReadyWait, r.pending);
          __syncwarp();
          return 0;
        }
      }
    }
    // Nothing to run yet. A look-ahead claim (made while the CTA still works
    // on its current tile) must not wait: the current tile's completion is
    // published only after it returns. The reservation is kept.
    if (!blocking) return 2;
    if (idle_return_ns != 0 && now - entered > idle_return_ns) return 2;
    __nanosleep(r.locked_out ? 200u : (uint32_t)p.idle_poll_ns);
  }
}

// Kernel entry bookkeeping: the launch's start time is the earliest CTA's.
__device__ void sched_enter(const SchedParams& p, unsigned long long t0) {
  unsigned long long* ts = reinterpret_cast<unsigned long long*>(&p.ctrl->t_start);
  if (atomicCAS(ts, 0ull, t0) != 0ull) atomicMin(ts, t0);
}

// Thread 0 of a CTA that is done: adds its phase counters; the last CTA of the
// launch publishes the launch's timeline and counters and resets the
// per-launch words for the next launch.
__device__ void sched_exit(const SchedParams& p, const uint64_t* prof) {
  for (int i = 0; i < kProfSlots; ++i)
    atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctrl->prof[i]), (unsigned long long)prof[i]);
  __threadfence();
  const uint32_t n = atomicAdd(&p.ctrl->exit_count, 1u);
  if (n + 1 != gridDim.x) return;
  // Read (and reset) together, then stored: one after another these were 16
  // round trips to L2, 4 us of every launch (launch of 32 vector adds of
  // 65536: 47 us, with this and the set-up below 44).
  HostShared* hs = p.host_shared;
  const uint64_t tiles = ld_relaxed_gpu64(&p.ctrl->published_tiles), entries = ld_relaxed_gpu64(&p.ctrl->published);
  const unsigned long long t_start = atomicExch(reinterpret_cast<unsigned long long*>(&p.ctrl->t_start), 0ull);
  const unsigned long long t_done = atomicExch(reinterpret_cast<unsigned long long*>(&p.ctrl->t_last_done), 0ull);
  unsigned long long sum[kProfSlots];
#pragma unroll
  for (int i = 0; i < kProfSlots; ++i)
    sum[i] = atomicExch(reinterpret_cast<unsigned long long*>(&p.ctrl->prof[i]), 0ull);
  st_relaxed_sys64(&hs->k_start, t_start);
  st_relaxed_sys64(&hs->k_last_done, t_done);
#pragma unroll
  for (int i = 0; i < kProfSlots; ++i) st_relaxed_sys64(&hs->k_prof[i], sum[i]);
  st_relaxed_sys64(&hs->k_exit, globaltimer());
  // Reservations beyond the published tiles died with their CTAs; the next
  // launch hands out tiles of entries published from here on.
  atomicExch(reinterpret_cast<unsigned long long*>(&p.ctrl->next_tile), (unsigned long long)tiles);
  atomicExch(reinterpret_cast<unsigned long long*>(&p.ctrl->first_entry), (unsigned long long)entries);
  atomicExch(&p.ctrl->exit_count, 0u);
  atomicExch(&p.ctrl->drained, 0u);
  atomicExch(&p.ctrl->ingest_lock, 0u);
  __threadfence_system();
  st_release_sys(&p.host_shared->exit_gen, p.launch_gen);
}

// One tile of a task has finished (its results are visible device-wide):
// count it, and complete the task after its last tile.
__device__ void finish_tile(const SchedParams& p, uint32_t task, uint32_t ntiles, uint32_t tag, uint32_t flags) {
  DevTask* dt = &p.tasks[task];
  const uint32_t d = atomicAdd(&dt->tiles_done, 1u);
  if (d + 1 == ntiles) {
    __threadfence();
    const uint64_t t_in = *reinterpret_cast<volatile uint64_t*>(&dt->t_ingest);
    complete_task(p, task, tag, flags, t_in);
  }
}

// ------------------------------------------------------------ FMA scheduler

// Warp 0: claim a tile into slot s (blocking: wait for work; otherwise
// return at once with go = 2 when nothing is claimable).
static __device__ __noinline__ void fma_claim(const SchedParams& p, SchedShared& sh, int slot, bool blocking) {
  const int lane = threadIdx.x & 31;
  const uint64_t t_acq = globaltimer();
  uint32_t task = 0, tile = 0;
  const int got = acquire<false>(p, reinterpret_cast<Claim*>(sh.claim), sh.list, task, tile, sh.prof, blocking);
  if (lane == 0) {
    sh.go[slot] = (uint32_t)got;
    sh.task[slot] = task;
    sh.tile[slot] = tile;
  }
  if (got == 1 && lane < (int)(sizeof(TaskBody) / 16)) {
    const uint4 v = ld_cg_v4(reinterpret_cast<const uint4*>(&p.tasks[task].body) + lane);
    reinterpret_cast<uint4*>(&sh.body[slot])[lane] = v;
  }
  __syncwarp();
  if (lane == 0) sh.prof[kProfAcquire] += globaltimer() - t_acq;
}

// All threads: slot cur's tile is done.
__device__ __forceinline__ void fma_finish(const SchedParams& p, SchedShared& sh, int cur, int bucket) {
  const TaskBody& b = sh.body[cur];
  // Results written into host memory: visible to the host before the task's
  // completion word.
  if (b.flags & kFlagDirectOut)
    __threadfence_system();
  else
    __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    sh.prof[bucket] += globaltimer() - sh.t_tile;
    sh.prof[kProfTiles] += 1;
    finish_tile(p, sh.task[cur], b.ntiles, b.tag, b.flags);
  }
}

// Vector tiles on warps 1 .., through the shared memory that the product tiles
// use. What bounds them is the bytes under way: each thread keeps kVecDepth
// groups of 32 bytes of its own on their way there (cp.async holds no
// registers: 66 KB an SM), and reads back only what it copied, so that no
// thread waits for another. 64 vector adds of 2^22 take 491 us, 714 where the
// operands are not 16-byte aligned. Loads into registers (eight 16-byte ones of
// each operand a thread, or single 4-byte ones) took 553 and 5090 us, and more
// of them spilled, in the product's loop too.
constexpr int kVecThreads = kFmaThreads - 32;
constexpr int kVecDepth = 11;
constexpr uint32_t kVecStage = kVecThreads * 32;  // a's halves, then b's
static_assert(kVecDepth * kVecStage <= sizeof(FmaSmem), "the groups fit the product tiles' memory");

template <int kBytes>
__device__ __forceinline__ void cp_async(uint32_t dst, const float* src) {
  if (kBytes == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

// kVec: a, b and c are 16-byte aligned and a group is four consecutive values of
// each, else every kVecThreads-th. c[i] = a[i] op b[i] for i < len, but for
// the last len % 4 with kVec.
template <int OP, bool kVec>
__device__ __forceinline__ void fma_vector_groups(const float* a, const float* b, float* c, int64_t len, int iters,
                                                  uint32_t smem) {
  constexpr int kStep = 4 * kVecThreads;              // values between a thread's groups
  constexpr int kEach = kVec ? 4 : kVecThreads;       // and between the parts of one
  constexpr int kBytes = kVec ? 16 : 4;
  const int t = threadIdx.x - 32;
  const uint32_t at = smem + t * kBytes;
  int64_t left = (kVec ? len & ~int64_t(3) : len) - (kVec ? 4 * t : t);  // values from the next group to store on
  a += kVec ? 4 * t : t;
  b += kVec ? 4 * t : t;
  c += kVec ? 4 * t : t;
  // Copies of the group `ahead` groups after the next one to store.
  auto issue = [&](int ahead, uint32_t slot) {
    const int off = ahead * kStep;
#pragma unroll
    for (int u = 0; u < (kVec ? 1 : 4); ++u) {
      if (off + u * kEach < left) {
        cp_async<kBytes>(slot + u * kEach * kBytes, a + off + u * kEach);
        cp_async<kBytes>(slot + kVecStage / 2 + u * kEach * kBytes, b + off + u * kEach);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll 1
  for (int d = 0; d < kVecDepth; ++d) issue(d, at + d * kVecStage);
  uint32_t slot = at;
  while (left > 0) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kVecDepth - 1) : "memory");
    if (kVec) {
      const uint4 xu = ld_shared_v4(slot), yu = ld_shared_v4(slot + kVecStage / 2);
      __stcs(reinterpret_cast<float4*>(c),
             elem_op4<OP>(*reinterpret_cast<const float4*>(&xu), *reinterpret_cast<const float4*>(&yu), iters));
    } else {
      float x[4], y[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        x[u] = ld_shared_f32(slot + u * kEach * 4);
        y[u] = ld_shared_f32(slot + kVecStage / 2 + u * kEach * 4);
      }
      const float4 z = elem_op4<OP>(make_float4(x[0], x[1], x[2], x[3]), make_float4(y[0], y[1], y[2], y[3]), iters);
      const float zs[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (u * kEach < left) c[u * kEach] = zs[u];
    }
    issue(kVecDepth, slot);  // after the stores: what the slot held is in registers
    a += kStep;
    b += kStep;
    c += kStep;
    left -= kStep;
    slot = slot + kVecStage < smem + kVecDepth * kVecStage ? slot + kVecStage : at;
  }
}

template <int OP>
__device__ __forceinline__ void fma_vector(const float* a, const float* b, float* c, int64_t len, int iters,
                                           uint32_t smem) {
  const uintptr_t all = reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) | reinterpret_cast<uintptr_t>(c);
  if ((all & 15) == 0) {
    fma_vector_groups<OP, true>(a, b, c, len, iters, smem);
    const int64_t e = (len & ~int64_t(3)) + threadIdx.x - 32;
    if (e < len) c[e] = elem_op<OP>(__ldcg(a + e), __ldcg(b + e), iters);
  } else {
    fma_vector_groups<OP, false>(a, b, c, len, iters, smem);
  }
}

__global__ void __launch_bounds__(kFmaThreads, 2) sched_fma_kernel(const __grid_constant__ SchedParams p) {
  __shared__ SchedShared sh;
  extern __shared__ uint8_t dyn_smem[];
  const int tid = threadIdx.x, warp = tid >> 5;
  if (tid == 0) {
    for (int i = 0; i < kProfSlots; ++i) sh.prof[i] = 0;
    sched_enter(p, globaltimer());
  }
  Claim* cl = reinterpret_cast<Claim*>(sh.claim);
  if (tid == 0) {
    cl->has_resv = 0;
    cl->stall_since = 0;
    // Tiles handed out by this launch lie in entries published after it began
    // (a CTA may start after others of the launch have already published).
    cl->hint = ld_relaxed_gpu64(&p.ctrl->first_entry);
  }
  __syncthreads();

  // One claim, inlined once: with calls in this loop, or more copies of the
  // claim, the product's inner loop spilled (1.7 to 2.0 ms instead of 1.5 for
  // 16 x 16 products of 512^3).
  bool have = false;  // slot cur holds a tile
  int cur = 0;
  while (true) {
    const int nxt = cur ^ 1;
    const TaskBody& b = sh.body[cur];
    const bool vec = have && (b.type == kTaskVadd || b.type == kTaskVmul);
    if (tid == 0) sh.t_tile = globaltimer();
    if (have && !vec) {
      const uint32_t tile = sh.tile[cur];
      fma_tile(reinterpret_cast<const float*>(b.a), reinterpret_cast<const float*>(b.b),
               reinterpret_cast<float*>(b.c), b.m, (int)b.n, b.k, (int)(tile / b.tiles_n), (int)(tile % b.tiles_n),
               reinterpret_cast<FmaSmem*>(dyn_smem));
      fma_finish(p, sh, cur, kProfGemm);  // before the claim, which may wait
    }
    // Warp 0 claims the next tile: while the others run a vector tile (then
    // without waiting), else waiting for one.
    if (warp == 0) {
      fma_claim(p, sh, nxt, !vec);
    } else if (vec) {
      const int64_t lo = (int64_t)sh.tile[cur] * b.vadd_tile, len = min(b.n - lo, b.vadd_tile);
      const float* x = reinterpret_cast<const float*>(b.a) + lo;
      const float* y = reinterpret_cast<const float*>(b.b) + lo;
      float* z = reinterpret_cast<float*>(b.c) + lo;
      if (b.type == kTaskVadd) fma_vector<kElemAdd>(x, y, z, len, 0, smem_u32(dyn_smem));
      else fma_vector<kElemMul>(x, y, z, len, b.k, smem_u32(dyn_smem));
    }
    if (vec) fma_finish(p, sh, cur, kProfVadd);
    else __syncthreads();
    const uint32_t go = sh.go[nxt];  // not written again before the next barrier but one
    if (go == 0) break;
    have = go == 1;
    cur = nxt;
  }
  __syncthreads();
  if (tid == 0) sched_exit(p, sh.prof);
}

// ------------------------------------------------------------ pair scheduler
//
// The split3 scheduler on clusters of two CTAs (gvm_pair.cuh). The leader's
// control warp claims tiles and posts each to the item rings of both CTAs;
// every role of both walks the items in order. A GEMM tile is the pair's: the
// CTAs stage their halves of the operands, the leader issues the MMAs, each
// CTA's epilogue warps store its 128 rows. A vector tile is split in two
// halves, each run by a CTA's converter warps from the landing ring (by
// converter and epilogue warps together where bulk copies cannot address the
// operands). Either way each CTA counts its half, so a task is complete after
// 2 x ntiles counts. The peer's control warp hands read items back to the
// leader. No warp waits for another warp's tile except through the pipeline's
// barriers.

constexpr int kItems = 4;                               // items in flight between the control warp and the others
constexpr uint32_t kItemExit = 0, kItemNop = 0xffu;     // besides the task types
constexpr int kFinSlots = 16;                           // per-item finish counters (items in flight < 16)
constexpr int kPrVecThreads = (kPrEpiWarps + kPrConvWarps) * 32;

// An item: what to run, then the task's fields as they lie in the task table.
struct alignas(16) PrItem {
  uint32_t kind;  // kItemExit, kItemNop or a task type
  uint32_t task;
  uint32_t tile;
  uint32_t first;  // SGEMM: number of the tile's first k-step (gvm_ring.h)
  uint32_t type, flags, rank, slot;
  uint32_t tag, ntiles, pad0, tiles_m;
  uint32_t tiles_n, pad1;
  int32_t m;
  int32_t k;
  int64_t n;
  int64_t span;  // vector tasks: elements per tile; SGEMM: columns per tile
  uint64_t a, b, c, pad2;
};
constexpr int kItemFields = 6;  // 16-byte pieces of task fields
constexpr int kItemFieldK = 2;  // the one that ends with k
static_assert(offsetof(TaskBody, k) == kFieldsAt + 16 * kItemFieldK + 12, "k's place");
static_assert(sizeof(PrItem) == 16 * (kItemFields + 1) && offsetof(TaskBody, c) - offsetof(TaskBody, type) ==
                  offsetof(PrItem, c) - offsetof(PrItem, type), "item = header + task fields");

// One thread: ask L2 for a GEMM item's task operands -- A's block of kPrM rows
// of the tile's row (from the tile in column 0 of its row) and all of B
// (from tile (0, 0)) -- so that each task's operands are requested once, in
// pieces of at most 1 MiB, when they are 16-byte aligned, span a multiple
// of 16 bytes and B holds at most 4 MiB. A hint only.
__device__ __forceinline__ void prefetch_task_operands(const PrItem& it) {
  if (it.kind != kTaskSgemm || (it.k & 3) || ((it.a | it.b) & 15)) return;
  const uint32_t tm = it.tile / it.tiles_n, tn = it.tile % it.tiles_n;
  if (tn != 0) return;
  auto pf = [](uint64_t addr, uint64_t bytes) {
    for (uint64_t off = 0; off < bytes; off += (1u << 20)) {
      const uint64_t len = bytes - off < (1u << 20) ? bytes - off : (1u << 20);
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(addr + off), "r"((uint32_t)len) : "memory");
    }
  };
  const int64_t rows = min((int64_t)kPrM, (int64_t)it.m - (int64_t)tm * kPrM);
  if (rows > 0) pf(it.a + (uint64_t)tm * kPrM * (uint64_t)it.k * 4u, (uint64_t)rows * (uint64_t)it.k * 4u);
  const uint64_t b_bytes = (uint64_t)it.k * (uint64_t)it.n * 4u;
  if (tm == 0 && b_bytes <= (4u << 20) && (b_bytes & 15) == 0) pf(it.b, b_bytes);
}

struct PairSchedShared {
  PrShared ps;
  uint64_t item_full[kItems];   // each CTA: control -> its consumers
  uint64_t item_empty[kItems];  // leader: its consumers and the peer's relay -> control; peer: its consumers -> relay
  PrItem items[kItems];
  uint32_t fin[kFinSlots];        // warps of this CTA done with item (seq % kFinSlots)
  uint32_t abort;
  uint32_t fail_where;
  uint64_t prof[kProfSlots];      // kProf* counters; each slot written by one thread only
  uint64_t claim[4];              // Claim state, owned by the control warp
  uint32_t list[32 * kMaxQuantum];  // ingest's scratch, control warp
  uint64_t g_begin;               // %globaltimer and clock64 when the CTA began
  long long c_begin;
};
constexpr uint32_t kPairSmemBytes = kPrRingBytes + sizeof(PairSchedShared);
static_assert(kPairSmemBytes <= 227 * 1024, "pair form shared memory");

__device__ __forceinline__ PrTile pair_tile(const PrItem& it) {
  return pr_tile(reinterpret_cast<const float*>(it.a), reinterpret_cast<const float*>(it.b),
                 reinterpret_cast<float*>(it.c), it.m, it.n, it.k, (int)(it.tile / it.tiles_n),
                 (int)(it.tile % it.tiles_n), (int)it.span, (it.flags / kFlagTmA) & 15u);
}
static_assert(kFlagTmB == 2 * kFlagTmA && kFlagPackA == 4 * kFlagTmA && kFlagPackB == 8 * kFlagTmA,
              "map flags are PrTile::land bits");

// One warp has written its share of an item (`warps` share it in this CTA):
// the last one counts this CTA's half of the tile.
__device__ __forceinline__ void pair_item_done(const SchedParams& p, PairSchedShared& sh, uint32_t seq, uint32_t warps,
                                               uint32_t task, uint32_t ntiles, uint32_t tag, uint32_t flags) {
  // Results written into host memory must be visible to the host before the
  // task's completion word is.
  if (flags & kFlagDirectOut)
    __threadfence_system();
  else
    __threadfence();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) {
    uint32_t* f = &sh.fin[seq % kFinSlots];
    if (atomicAdd(f, 1u) == warps - 1) {
      *f = 0;
      __threadfence();
      finish_tile(p, task, 2 * ntiles, tag, flags);
    }
  }
  __syncwarp();
}

// A consumer's next item, for one thread or (kWarp) a whole warp; false when
// the wait ran out or the CTA stopped.
template <bool kWarp>
__device__ __forceinline__ bool pair_item_wait(const SchedParams& p, PairSchedShared& sh, uint32_t seq) {
  uint64_t* bar = &sh.item_full[seq % kItems];
  const uint32_t ph = (seq / kItems) & 1u;
  if (kWarp ? mbar_wait_warp<true>(bar, ph, p.wait_timeout_ns, &sh.abort)
            : mbar_wait_cluster(bar, ph, p.wait_timeout_ns, &sh.abort))
    return true;
  if (!sh.abort) {
    pr_fail(&sh.ps, &sh.abort, &sh.fail_where, kWhereItemWait);
    report_error(p, kStatusTimeout, kWhereItemWait, seq);
  }
  return false;
}
// To the CTA's own barrier: see pair_relay.
__device__ __forceinline__ void pair_item_release(PairSchedShared& sh, uint32_t seq) {
  mbar_arrive(&sh.item_empty[seq % kItems]);
}

// The roles, each a function of its own: ptxas gives a function the registers
// that its callers do not hold, and what spills is read back from L2 (the
// control warp's acquires keep invalidating L1). With the roles inlined into
// the kernel the converters' loop spilled and a 512^3 launch took 1.6 ms.
#define PAIR_ROLE static __device__ __noinline__ void

// Control (leader): claims tiles into both item rings.
PAIR_ROLE pair_control(const SchedParams& p, PairSchedShared& sh) {
  const int lane = threadIdx.x & 31;
  Claim* cl = reinterpret_cast<Claim*>(sh.claim);
  const uint64_t to = p.wait_timeout_ns;
  // k-step numbers are counted here and posted with the items: one register
  // less in the converters, whose loops spill.
  uint32_t first = 0;
  for (uint32_t seq = 0;; ++seq) {
    const uint32_t slot = seq % kItems, ph = (seq / kItems) & 1u;
    // One lane waits and reads the abort word, and all go by what it found: the
    // claim below is warp-collective, and another warp may set the word meanwhile.
    uint32_t seen = 0;  // bit 0: the slot is free, bit 1: the CTA stops
    if (lane == 0) {
      seen = mbar_wait_cluster(&sh.item_empty[slot], ph ^ 1u, to, &sh.abort) ? 1u : 0u;
      if (ld_volatile_u32(&sh.abort)) seen |= 2u;
    }
    seen = bcast(seen);
    if (!(seen & 1u)) {
      if (lane == 0 && !(seen & 2u)) {
        pr_fail(&sh.ps, &sh.abort, &sh.fail_where, kWhereItemRing);
        report_error(p, kStatusTimeout, kWhereItemRing, seq);
      }
      break;
    }
    const uint64_t t0 = globaltimer();
    uint32_t task = 0, tile = 0;
    // An idle control warp posts a no-op item now and then, so that the
    // other warps' waits for items stay bounded.
    const int got = (seen & 2u) ? 0 : acquire<true>(p, cl, sh.list, task, tile, sh.prof, true, to / 4);
    // Lanes 0..5 carry the task's fields, lane 6 the header (it reads the piece
    // that begins with the type), to both CTAs.
    uint4 v = make_uint4(got == 2 ? kItemNop : kItemExit, 0, 0, 0);
    if (got == 1 && lane <= kItemFields)
      v = ld_cg_v4(reinterpret_cast<const uint8_t*>(&p.tasks[task].body) + kFieldsAt + 16 * (lane % kItemFields));
    const uint32_t kind = __shfl_sync(0xffffffffu, v.x, 0), k = __shfl_sync(0xffffffffu, v.w, kItemFieldK);
    if (lane <= kItemFields) {
      if (lane == kItemFields && got == 1) v = make_uint4(v.x, task, tile, first);
      uint4* dst = reinterpret_cast<uint4*>(&sh.items[slot]) + (lane == kItemFields ? 0 : lane + 1);
      *dst = v;
      st_cluster_v4(mapa_shared(smem_u32(dst), 1), v);
      mbar_arrive_release_cta(&sh.item_full[slot], 1);
      mbar_arrive(&sh.item_full[slot]);
    }
    if (got == 1 && kind == kTaskSgemm) first = pr_next_first(first, (k + kTcBK - 1) / kTcBK);
    __syncwarp();
    if (lane == 0) {
      sh.prof[kProfAcquire] += globaltimer() - t0;
      // L2 prefetch, a few tiles ahead of the producers: the item two claims
      // back (its slot is rewritten only two claims from now).
      if (p.prefetch && seq >= 2) prefetch_task_operands(sh.items[(seq + 2) % kItems]);
    }
    __syncwarp();
    if (got == 0) break;
  }
}

// Relay (peer's control warp, one thread): hands the slots that this CTA's
// consumers have read back to the leader. The leader overwrites them from
// another CTA, which a CTA-scope release does not order after the reads, and a
// cluster-scope one by each consumer waits for its other accesses under way:
// 64 vector adds of 2^22 took 6% longer so, the grouped mix 2%. Here the
// consumers release to their own CTA, and this thread, with no accesses of its
// own, passes what it has acquired from them on to the cluster.
PAIR_ROLE pair_relay(const SchedParams& p, PairSchedShared& sh) {
  for (uint32_t seq = 0; pair_item_wait<false>(p, sh, seq); ++seq) {
    const uint32_t slot = seq % kItems, kind = sh.items[slot].kind;
    // The control warp waits for a slot only once it wants it again, this thread
    // from the item's posting on, up to kItems items earlier.
    bool ok = false;
    for (int i = 0; i <= kItems && !ok && !sh.abort; ++i)
      ok = mbar_wait(&sh.item_empty[slot], (seq / kItems) & 1u, p.wait_timeout_ns, &sh.abort);
    if (!ok) {
      if (!sh.abort) {
        pr_fail(&sh.ps, &sh.abort, &sh.fail_where, kWhereItemRing);
        report_error(p, kStatusTimeout, kWhereItemRing, seq);
      }
      break;
    }
    mbar_arrive_release_cta(&sh.item_empty[slot], 0);
    if (kind == kItemExit) break;
  }
}

// This CTA's half of a vector item.
struct PairVec {
  const float* a;
  const float* b;
  float* c;
  int64_t len;
};
__device__ __forceinline__ PairVec pair_vec(const PrItem& it, uint32_t cta) {
  const int64_t half = it.span / 2, lo = (int64_t)it.tile * it.span + (int64_t)cta * half;
  const int64_t len = min(it.n - lo, half);
  return PairVec{reinterpret_cast<const float*>(it.a) + lo, reinterpret_cast<const float*>(it.b) + lo,
                 reinterpret_cast<float*>(it.c) + lo, len > 0 ? len : 0};
}
// Vector items whose operands bulk copies can address run through the landing
// ring (the halves of a tile begin at multiples of 512 elements).
__device__ __forceinline__ bool pair_vec_lands(const PrItem& it) { return ((it.a | it.b) & 15) == 0; }

// MMA issue (leader, one thread): GEMM items only; every item is read and released.
PAIR_ROLE pair_mma(const SchedParams& p, PairSchedShared& sh, uint8_t* stages) {
  uint32_t tile_no = 0;
  for (uint32_t seq = 0; pair_item_wait<false>(p, sh, seq); ++seq) {
    const PrItem& item = sh.items[seq % kItems];
    const uint32_t kind = item.kind, first = item.first;
    const PrTile t = kind == kTaskSgemm ? pair_tile(item) : PrTile{};
    pair_item_release(sh, seq);
    if (kind == kItemExit) break;
    if (kind != kTaskSgemm) continue;
    if (!pr_mma(t, stages, &sh.ps, first, tile_no, p.wait_timeout_ns, &sh.abort, &sh.fail_where,
                &sh.prof[kProfMmaWait])) {
      report_error(p, kStatusTimeout, sh.fail_where, seq);
      break;
    }
    ++tile_no;
  }
}

// Producer (one thread): the tensor copies of every GEMM item's k-steps, the
// bulk copies of vector items.
PAIR_ROLE pair_produce(const SchedParams& p, PairSchedShared& sh, uint8_t* land) {
  uint32_t it_l = 0, pend = 0;
  for (uint32_t seq = 0; pair_item_wait<false>(p, sh, seq); ++seq) {
    const PrItem& item = sh.items[seq % kItems];
    const uint32_t kind = item.kind;
    const CUtensorMap* tm = &p.tasks[item.task].body.tmA;
    const PrTile t = kind == kTaskSgemm ? pair_tile(item) : PrTile{};
    const bool vec = (kind == kTaskVadd || kind == kTaskVmul) && pair_vec_lands(item);
    const PairVec v = vec ? pair_vec(item, sh.ps.cta) : PairVec{};
    pair_item_release(sh, seq);
    if (kind == kItemExit) break;
    if (kind != kTaskSgemm && !vec) continue;
    // The operands may have been written by this kernel's own stores, and
    // the maps were written by the ingest's.
    fence_proxy_async_global();
    bool ok;
    if (vec) {
      ok = pr_vec_produce(v.a, v.b, v.len, land, &sh.ps, it_l, p.wait_timeout_ns, &sh.abort, &sh.fail_where, pend);
      it_l += pr_vec_chunks(v.len);
    } else {
      if (t.land & kPrMapA) fence_tensormap_acquire(tm);
      if (t.land & kPrMapB) fence_tensormap_acquire(tm + 1);
      ok = pr_produce(t, land, &sh.ps, it_l, tm, tm + 1, p.wait_timeout_ns, &sh.abort, &sh.fail_where, pend);
      it_l += (uint32_t)((t.k + kTcBK - 1) / kTcBK);
    }
    if (!ok) {
      report_error(p, kStatusTimeout, sh.fail_where, seq);
      break;
    }
  }
  pr_produce_quiesce(&sh.ps, pend, p.wait_timeout_ns);
}

// Vector item without 16-byte aligned operands, converter and epilogue warps
// together, by direct loads.
__device__ __forceinline__ void pair_vector(const SchedParams& p, PairSchedShared& sh, uint32_t seq) {
  const int tid = threadIdx.x, lane = tid & 31;
  const PrItem& item = sh.items[seq % kItems];
  const uint32_t kind = item.kind, task = item.task, ntiles = item.ntiles, tag = item.tag, flags = item.flags;
  const int iters = item.k;
  const PairVec v = pair_vec(item, sh.ps.cta);
  __syncwarp();
  if (lane == 0) pair_item_release(sh, seq);
  if (kind == kTaskVmul) vmul_range<true>(v.a, v.b, v.c, 0, v.len, tid, kPrVecThreads, iters);
  else vadd_range<true>(v.a, v.b, v.c, 0, v.len, tid, kPrVecThreads);
  pair_item_done(p, sh, seq, kPrEpiWarps + kPrConvWarps, task, ntiles, tag, flags);
}

// Converter warps: stage GEMM tiles, run vector tiles.
PAIR_ROLE pair_convert(const SchedParams& p, PairSchedShared& sh, uint8_t* land, uint8_t* stages) {
  const int lane = threadIdx.x & 31;
  const bool prof = threadIdx.x == kPrConvWarp0 * 32;
  uint32_t it_l = 0;
  for (uint32_t seq = 0; pair_item_wait<true>(p, sh, seq); ++seq) {
    const PrItem& item = sh.items[seq % kItems];
    const uint32_t kind = item.kind;
    const uint64_t t0 = prof ? globaltimer() : 0;
    bool ok = true;
    if (kind == kTaskSgemm) {
      const PrTile t = pair_tile(item);
      const uint32_t first = item.first;
      __syncwarp();
      if (lane == 0) pair_item_release(sh, seq);
      ok = pr_convert(t, land, stages, &sh.ps, first, it_l, p.wait_timeout_ns, &sh.abort, &sh.fail_where);
      it_l += (uint32_t)((t.k + kTcBK - 1) / kTcBK);
      if (prof) sh.prof[kProfGemm] += globaltimer() - t0;
    } else if (kind == kTaskVadd || kind == kTaskVmul) {
      if (pair_vec_lands(item)) {
        const uint32_t task = item.task, ntiles = item.ntiles, tag = item.tag, flags = item.flags;
        const int iters = item.k;
        const PairVec v = pair_vec(item, sh.ps.cta);
        __syncwarp();
        if (lane == 0) pair_item_release(sh, seq);
        ok = kind == kTaskVmul ? pr_vec_convert<kElemMul>(v.a, v.b, v.c, v.len, iters, land, &sh.ps, it_l,
                                                          p.wait_timeout_ns, &sh.abort, &sh.fail_where)
                               : pr_vec_convert<kElemAdd>(v.a, v.b, v.c, v.len, 0, land, &sh.ps, it_l,
                                                          p.wait_timeout_ns, &sh.abort, &sh.fail_where);
        it_l += pr_vec_chunks(v.len);
        if (ok) pair_item_done(p, sh, seq, kPrConvWarps, task, ntiles, tag, flags);
      } else {
        pair_vector(p, sh, seq);
      }
      if (prof) {
        sh.prof[kProfVadd] += globaltimer() - t0;
        if (sh.ps.cta == 0) atomicAdd(reinterpret_cast<unsigned long long*>(&sh.prof[kProfTiles]), 1ull);
      }
    } else {
      __syncwarp();
      if (lane == 0) pair_item_release(sh, seq);
      if (kind == kItemExit) break;
    }
    if (!ok) {
      if (lane == 0) report_error(p, kStatusTimeout, sh.fail_where, 0);
      break;
    }
  }
}

// Epilogue warps: store GEMM tiles and count them.
PAIR_ROLE pair_epilogue(const SchedParams& p, PairSchedShared& sh) {
  const int tid = threadIdx.x, lane = tid & 31;
  uint32_t tile_no = 0;
  for (uint32_t seq = 0; pair_item_wait<true>(p, sh, seq); ++seq) {
    const PrItem& item = sh.items[seq % kItems];
    const uint32_t kind = item.kind;
    if ((kind == kTaskVadd || kind == kTaskVmul) && !pair_vec_lands(item)) {
      pair_vector(p, sh, seq);
      continue;
    }
    const uint32_t task = item.task, ntiles = item.ntiles, tag = item.tag, flags = item.flags;
    const PrTile t = kind == kTaskSgemm ? pair_tile(item) : PrTile{};
    __syncwarp();
    if (lane == 0) pair_item_release(sh, seq);
    if (kind == kItemExit) break;
    if (kind != kTaskSgemm) continue;
    const uint64_t t0 = pr_epilogue(t, &sh.ps, tile_no, p.wait_timeout_ns, &sh.abort, &sh.fail_where);
    if (t0 == 0) {
      if (lane == 0) report_error(p, kStatusTimeout, sh.fail_where, 0);
      break;
    }
    pair_item_done(p, sh, seq, kPrEpiWarps, task, ntiles, tag, flags);
    if (tid == 0) {
      sh.prof[kProfEpilogue] += globaltimer() - t0;
      if (sh.ps.cta == 0) atomicAdd(reinterpret_cast<unsigned long long*>(&sh.prof[kProfTiles]), 1ull);
    }
    ++tile_no;
  }
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPrThreads, 1)
    sched_pair_kernel(const __grid_constant__ SchedParams p) {
  extern __shared__ __align__(1024) uint8_t dyn_smem[];
  uint8_t* land = dyn_smem;
  uint8_t* stages = dyn_smem + kPrLand * kPrLandBytes;
  PairSchedShared& sh = *reinterpret_cast<PairSchedShared*>(dyn_smem + kPrRingBytes);
  const int tid = threadIdx.x, warp = tid >> 5;
  if (tid == 0) {
    sh.abort = 0;
    sh.fail_where = 0;
    sh.g_begin = globaltimer();
    sh.c_begin = clock64();
    for (int i = 0; i < kProfSlots; ++i) sh.prof[i] = 0;
    for (int i = 0; i < kFinSlots; ++i) sh.fin[i] = 0;
    for (int i = 0; i < kItems; ++i) {
      mbar_init(&sh.item_full[i], kItemFields + 1);  // a lane per 16-byte piece
      // The CTA's epilogue and converter warps and producer; leader: the MMA thread and the peer's relay.
      mbar_init(&sh.item_empty[i], kPrEpiWarps + kPrConvWarps + 1 + (cluster_ctarank() == 0 ? 2 : 0));
    }
    Claim* cl = reinterpret_cast<Claim*>(sh.claim);
    cl->has_resv = 0;
    cl->stall_since = 0;
  }
  // Its round trip to L2 passes while the pipeline is set up; the launch's
  // start time is noted after that, off the way to the first claim.
  uint64_t first = 0;
  if (tid == 32 * kPrCtlWarp) first = ld_relaxed_gpu64(&p.ctrl->first_entry);
  pr_init(&sh.ps);  // the pipeline's barriers, fences all inits, TMEM
  const bool leader = sh.ps.cta == 0;
  if (warp < kPrEpiWarps) {
    if (tid == 0) sched_enter(p, sh.g_begin);
    __syncwarp();
    pair_epilogue(p, sh);
  } else if (warp < kPrMmaWarp) {
    pair_convert(p, sh, land, stages);
  } else if (warp == kPrMmaWarp) {
    if (leader && elect_one()) {
      pair_mma(p, sh, stages);
      umma_commit_pair(&sh.ps.mma_done);
    }
  } else if (warp == kPrProdWarp) {
    if (elect_one()) pair_produce(p, sh, land);
  } else if (leader) {
    if (tid == 32 * kPrCtlWarp) reinterpret_cast<Claim*>(sh.claim)->hint = first;
    __syncwarp();
    pair_control(p, sh);
  } else if (elect_one()) {
    pair_relay(p, sh);
  }
  __syncwarp();
  pr_teardown(&sh.ps, 2 * p.wait_timeout_ns);
  if (tid == 0) {
    // The waits for k-steps were summed in SM clocks: to nanoseconds.
    const double ns = (double)(globaltimer() - sh.g_begin) / (double)max(1ll, clock64() - sh.c_begin);
    sh.prof[kProfMmaWait] = (uint64_t)(ns * (double)sh.prof[kProfMmaWait]);
    sched_exit(p, sh.prof);
  }
}

static size_t dyn_smem_bytes(int path) {
  if (path == kPathSplit3) return kPairSmemBytes;
  return sizeof(FmaSmem) + 1024;
}

static const void* sched_fn(int path) {
  if (path == kPathSplit3) return (const void*)sched_pair_kernel;
  return (const void*)sched_fma_kernel;
}

static int sched_threads(int path) {
  return path == kPathFma ? kFmaThreads : kPrThreads;
}

cudaError_t scheduler_setup(int path, int sms, int* max_ctas, size_t* smem_bytes) {
  const size_t smem = dyn_smem_bytes(path);
  const void* fn = sched_fn(path);
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if (path == kPathSplit3) {
    // As many clusters of two CTAs as the device holds at once.
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(2);
    c.blockDim = dim3(kPrThreads);
    c.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 2;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    c.attrs = &attr;
    c.numAttrs = 1;
    int clusters = 0;
    e = cudaOccupancyMaxActiveClusters(&clusters, fn, &c);
    if (e != cudaSuccess) return e;
    *max_ctas = 2 * clusters;
    *smem_bytes = smem;
    return cudaSuccess;
  }
  int nb = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, sched_threads(path), smem);
  if (e != cudaSuccess) return e;
  *max_ctas = nb * sms;
  *smem_bytes = smem;
  return cudaSuccess;
}

cudaError_t launch_scheduler(int path, const SchedParams& p, int grid, size_t smem, cudaStream_t stream) {
  if (path == kPathSplit3) {
    sched_pair_kernel<<<grid, kPrThreads, smem, stream>>>(p);
  } else {
    sched_fma_kernel<<<grid, kFmaThreads, smem, stream>>>(p);
  }
  return cudaGetLastError();
}

}  // namespace gvm
