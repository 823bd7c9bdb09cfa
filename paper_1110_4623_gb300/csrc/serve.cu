// Persistent serving loop with continuous batching, built on the library's own ticket lock and
// ticket-window semaphore (the paper motivates its primitives with task queues, Section 1, and
// names hardware enqueue/dequeue as a wish, Section 7).
//
// The host publishes requests into a ring of 16-byte entries (each entry carries its sequence
// number twice, one copy in each of its two 8-byte halves, each half written with one store).
// The ring is caller memory: pinned host memory, which the admitters poll across the host
// link, or managed memory placed in device memory, which the host writes in place and the
// admitters poll through L2.  Inside one co-resident
// launch:
//   * admitter blocks admit a batch of requests at a time, one per warp: they take the batch's
//     request indices with one acquisition of the ring's ticket lock, and each warp waits on the
//     admission semaphore (n = number of in-flight slots) for its request's permit, waits for
//     its entry to appear, claims a free slot and publishes the request in it (release store of
//     the slot's claim word);
//   * every other block claims chunks of any active slot (fetch-and-add on the slot's claim
//     word), sums the chunks' int32 values in int64 (with a backlog, a bounded run of one
//     request's), and adds its partial to the slot's accumulator; the block that finishes a
//     request writes the result and a completion flag into pinned host memory, frees the
//     slot and posts the semaphore.
// Requests that arrive while others run are admitted as slots free up and their chunks run
// side by side with older requests' chunks.  Every wait is bounded (the object timeouts, or
// the loop's own deadline) and the host's shutdown word ends the loop.
//
// The per-request-launch baseline runs the same chunked segmented sum as one kernel launch
// per request and completes it the same way (result and flag in pinned host memory).
#include <pthread.h>
#include <stddef.h>
#include <sched.h>
#include <string.h>
#include <unistd.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <thread>
#include <vector>

#include "common.cuh"

using namespace gsync_impl;
namespace ptx = gsync::ptx;

namespace {

constexpr int kThreads = 256;
// Ring entries sit one per 128-byte line, so the host writing entry q never touches a line
// that an admitter polls for another entry.
constexpr size_t kRingStride = 128;
static_assert(sizeof(gsync_serve_req) == 16 && offsetof(gsync_serve_req, seq) == 0 &&
                  offsetof(gsync_serve_req, len) == 4 && offsetof(gsync_serve_req, off) == 8 &&
                  offsetof(gsync_serve_req, seq_check) == 12,
              "the producer writes an entry as two 8-byte halves {seq, len} and {off, seq_check}");
static_assert(__BYTE_ORDER__ == __ORDER_LITTLE_ENDIAN__, "the entry halves are packed little-endian");
// The active mask is kept in kMaskCopies copies on separate lines (set and cleared in all,
// read from one per worker) to spread the workers' polling.
constexpr uint32_t kMaskCopies = 4;
// Active slots from which a worker goes on with the chunks of the request it has: at 1e6 req/s
// about seven requests are in flight, a drained backlog keeps most slots active.
constexpr int kBacklog = 8;
// ... and the most chunks it takes of one request before it looks at the others again: a worker that
// stayed until the request had no more left was lost to the short requests beside a long one (64
// slots, 3 workers, 600 requests of one chunk beside one of 30,000: the short ones done after 12.3 ms
// instead of 0.9).  At 16 a backlog of 3000 requests in chunks of 2048 takes as long as without a
// limit (3.58 and 3.59 ms), at 8 as well (3.61), at 4 3.72.
constexpr uint32_t kKeep = 16;

struct Slot {  // one 128-byte line
  // The claim word: chunk count << 32 | next chunk to hand out.  Only ever read, added to and
  // published as one 64-bit word, so a claim always sees the count of the request whose chunk it
  // took.  A slot with no request has no chunk left (never used: 0 of 0; finished: past the last).
  uint64_t claim;
  uint32_t done_chunks;
  uint32_t id;
  int64_t off;
  int64_t len;
  unsigned long long acc;
  uint32_t pad[22];
};
static_assert(sizeof(Slot) == 128, "one line per slot");

struct Args {
  const gsync_serve_req* ring;  // device view of the host ring
  uint32_t ring_mask;
  const uint32_t* shutdown;  // device view (host writes)
  uint32_t* dev_shutdown;    // device copy of the shutdown word, set by an admitter (own line)
  int64_t* res;              // device view of host results
  uint32_t* done;            // device view of host completion flags
  const int32_t* pool;
  uint32_t* ring_lock;       // gsync mutex (TICKET)
  uint32_t* admit_sem;       // gsync semaphore (WINDOW), n = nslots
  Slot* slots;
  uint32_t* active_mask;     // one bit per slot (nslots <= 64)
  unsigned long long* busy;  // one bit per slot that a lane has claimed and no worker has freed yet
  uint32_t* stats;           // [0] admitted, [32] chunks, [64] completed (own lines)
  uint32_t* status;
  unsigned long long* trace;  // optional per-request timestamps (4 per request)
  uint32_t nslots, admitters, chunk_elems;
  uint32_t lanes;            // admission lanes per admitter block (warps 0 .. lanes - 1)
  uint64_t timeout_ns;
};

__device__ __forceinline__ uint32_t ld_acquire_sys(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.sys.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// Two 8-byte accesses, each single-copy atomic, in no set order: the halves of a ring entry.  (A
// vector of four words would be four accesses, and a half's number could be newer than its value.)
__device__ __forceinline__ void ld_acquire_sys_v2(const void* p, uint64_t& lo, uint64_t& hi) {
  asm volatile("ld.acquire.sys.global.v2.u64 {%0, %1}, [%2];" : "=l"(lo), "=l"(hi) : "l"(p) : "memory");
}
__device__ __forceinline__ void st_release_sys(uint32_t* p, uint32_t v) {
  asm volatile("st.release.sys.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void st_relaxed_sys(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.sys.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void st_relaxed_sys_s64(int64_t* p, int64_t v) {
  asm volatile("st.relaxed.sys.global.s64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// This thread's share of the int64 sum of pool[a, b): 16-byte streaming loads over the aligned
// middle, eight of them in flight per thread (issued before any is added; the last, partial
// pass -- every request's last chunk -- too, with the loads past the end predicated off),
// scalars at the ends.
__device__ __forceinline__ long long thread_sum(const int32_t* pool, int64_t a, int64_t b) {
  constexpr int kInFlight = 8;
  long long s = 0;
  int64_t a4 = (a + 3) & ~(int64_t)3;
  if (a4 > b) a4 = b;
  const int64_t b4 = a4 + ((b - a4) & ~(int64_t)3);
  for (int64_t i = a + threadIdx.x; i < a4; i += blockDim.x) s += pool[i];
  const int4* v = reinterpret_cast<const int4*>(pool + a4);
  const int64_t nv = (b4 - a4) >> 2;
  const int64_t step = (int64_t)blockDim.x * kInFlight;
  int64_t i = threadIdx.x;
  for (; i + (kInFlight - 1) * (int64_t)blockDim.x < nv; i += step) {
    int4 x[kInFlight];
#pragma unroll
    for (int k = 0; k < kInFlight; ++k) x[k] = __ldcs(v + i + k * (int64_t)blockDim.x);
#pragma unroll
    for (int k = 0; k < kInFlight; ++k) s += (long long)x[k].x + x[k].y + x[k].z + x[k].w;
  }
  if (i < nv) {  // fewer than kInFlight left for this thread: issue them all before adding
    int4 x[kInFlight];
#pragma unroll
    for (int k = 0; k < kInFlight; ++k) {
      const int64_t j = i + k * (int64_t)blockDim.x;
      x[k] = j < nv ? __ldcs(v + j) : make_int4(0, 0, 0, 0);
    }
#pragma unroll
    for (int k = 0; k < kInFlight; ++k) s += (long long)x[k].x + x[k].y + x[k].z + x[k].w;
  }
  for (int64_t i = b4 + threadIdx.x; i < b; i += blockDim.x) s += pool[i];
  return s;
}

// Sum of the threads' shares, valid in thread 0.
__device__ __forceinline__ long long block_reduce(long long s) {
  __shared__ long long red[kThreads / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  long long t = 0;
  if (threadIdx.x == 0)
    for (uint32_t w = 0; w < (blockDim.x + 31) / 32; ++w) t += red[w];
  __syncthreads();
  return t;
}

__device__ __forceinline__ uint64_t atom_add_acquire_u64(uint64_t* p, uint64_t v) {
  uint64_t r;
  asm volatile("atom.acquire.gpu.global.add.u64 %0, [%1], %2;" : "=l"(r) : "l"(p), "l"(v) : "memory");
  return r;
}

// Thread 0: claims one chunk of a slot, or returns false.  A look comes first: only a slot with
// chunks left is worth a claim.  The claim is one fetch-and-add on the claim word, so racing
// workers each get a distinct chunk in one round trip, with the chunk count of the request it
// belongs to: of the one looked at, or of a newer one that took the slot since, and is served
// instead.  A claim past the count is an over-claim and is dropped (the count of a later request
// overwrites it; at most one per worker and request, far from the word's upper half).  A chunk
// that is claimed and not yet counted done keeps the slot with its request.  The acquire belongs
// to the claim, which reads the publication of the very request that it returns.
__device__ __forceinline__ bool claim_chunk(Slot* slot, uint32_t& chunk, uint32_t& nchunks) {
  const uint64_t look = ptx::ld_relaxed_u64(&slot->claim);
  if ((uint32_t)look >= (uint32_t)(look >> 32)) return false;
  const uint64_t v = atom_add_acquire_u64(&slot->claim, 1ull);
  chunk = (uint32_t)v;
  nchunks = (uint32_t)(v >> 32);
  return chunk < nchunks;
}

// Barrier over the admission lanes' warps of an admitter block (its other warps have left).
__device__ __forceinline__ void lanes_sync(uint32_t lanes) {
  __syncwarp();
  asm volatile("barrier.sync 1, %0;" ::"r"(lanes * 32u) : "memory");
}

// Thread 0 of an admitter: the next batch of ring indices, one for each lane.  The ring lock's
// tickets are handed out in order from 0, one per acquisition, so ticket t stands for the indices
// t * lanes .. + lanes - 1: the holder needs no head word and releases the lock at once, and as
// the lock hands on nothing but the ticket itself, the release needs no fence.
__device__ __forceinline__ bool take_indices(const Args& a, const gsync::MutexRef& lock, uint32_t& head) {
  if (ptx::ld_relaxed(a.dev_shutdown)) return false;
  const gsync::Token t = gsync::mutex_lock_thread<GSYNC_MUTEX_TICKET>(lock);
  if (t.status != GSYNC_OK) {
    record_status(a.status, t.status);
    return false;
  }
  ptx::st_relaxed(lock.turn(), t.ticket + 1u);
  head = t.ticket * a.lanes;
  return true;
}

// The shutdown word that the host sets, looked at by one of the lanes and passed on to all.
__device__ __forceinline__ bool host_shutdown(const Args& a) {
  if (!ld_acquire_sys(a.shutdown)) return false;
  ptx::st_release(a.dev_shutdown, 1u);
  return true;
}

// One lane: waits for a permit of the admission semaphore.  Every request takes one permit and one
// index, so the index is also its ticket of the window: request h enters once h - nslots + 1
// requests have completed.  Each lane enters by itself, so a request that takes long keeps one
// slot from the others, and not the batch behind it (a batch that entered with its last ticket waited
// for the whole one before with slots = lanes: 8 slots, 1 admitter, 7 of 8 slots empty beside a long
// request); and permits go out in the order of the ring, also where the ring is shorter than the
// indices taken.  False to stop.
__device__ __forceinline__ bool wait_permit(const Args& a, const gsync::SemRef& s, uint32_t h) {
  gsync::Waiter w;
  uint32_t polls = 0;
  for (;;) {
    const uint32_t turn = ptx::ld_acquire(s.word(2));
    if (gsync::after(turn + s.n, h)) return true;
    // the bound of one permit's wait, for each of the batch that a lane may wait behind
    if (int rc = w.tick(s.timeout_ns * a.lanes, s.abort_word())) {
      record_status(a.status, rc);
      return false;
    }
    ++polls;
    if ((polls & 7u) == 0u && ptx::ld_relaxed(a.dev_shutdown)) return false;
    if ((polls & 255u) == 0u && host_shutdown(a)) return false;
    const uint32_t ns = (h - (turn + s.n) + 1u) * s.bo.min_ns;
    gsync::sleep_to_poll(ns, s.bo.max_ns);
  }
}

// Claims a slot whose bit is clear in the busy word, h mod nslots if that one is free.  The atomic
// that sets a bit also returns the word, so a lane that loses a bit picks its next one from there
// (a walk over the slots' own state words pays a round trip for each busy slot it meets).  The
// permit guarantees a free slot, but not which, so this only ends without one at the deadline.
constexpr uint32_t kNoSlot = 0xFFFFFFFFu;
__device__ __forceinline__ uint32_t claim_slot(const Args& a, uint32_t h) {
  const uint64_t all = a.nslots == 64u ? ~0ull : (1ull << a.nslots) - 1ull;
  uint32_t s = h % a.nslots;
  uint64_t deadline = 0;
  for (;;) {
    const uint64_t bit = 1ull << s;
    uint64_t old;
    asm volatile("atom.acquire.gpu.global.or.b64 %0, [%1], %2;" : "=l"(old) : "l"(a.busy), "l"(bit) : "memory");
    if (!(old & bit)) return s;
    uint64_t free;
    while ((free = ~old & all) == 0) {  // the permit came before the slot's bit: it is on its way
      const uint64_t now = ptx::globaltimer();
      if (deadline == 0) deadline = now + a.timeout_ns;
      if (now > deadline) return kNoSlot;
      old = ptx::ld_relaxed_u64((const uint64_t*)a.busy);
    }
    // The r-th free bit, r by the request: lanes that lost the same bit part ways here (the next
    // free bit for all of them sent a batch's lanes at one bit again and again, 7.3 us to publish
    // a request under load against 1.9).
    uint32_t r = h % (uint32_t)__popcll(free);
    while (r--) free &= free - 1u;
    s = (uint32_t)__ffsll((long long)free) - 1u;
  }
}

// After a fence that orders the request's last use of the slot.
__device__ __forceinline__ void free_slot(const Args& a, uint32_t s) {
  asm volatile("red.relaxed.gpu.global.and.b64 [%0], %1;" ::"l"(a.busy), "l"(~(1ull << s)) : "memory");
}
// The slot's last chunk is handed out: it has no more work to find, so it leaves the active
// mask (it cannot be reused before that chunk completes).
__device__ __forceinline__ void retire_slot(const Args& a, uint32_t s) {
  for (uint32_t k = 0; k < kMaskCopies; ++k) atomicAnd(&a.active_mask[32u * k + (s >> 5)], ~(1u << (s & 31)));
}

// One lane: waits for a permit and for ring entry h (seq == seq_check == h + 1), claims a free slot
// and publishes the request in it.  False to stop (shutdown, or a wait that ran out).
__device__ __forceinline__ bool admit(const Args& a, const gsync::SemRef& sem, uint32_t h) {
  const gsync_serve_req* e = (const gsync_serve_req*)((const char*)a.ring + (size_t)(h & a.ring_mask) * kRingStride);
  if (!wait_permit(a, sem, h)) return false;
  uint64_t lo, hi;  // seq | len << 32 and off | seq_check << 32
  uint32_t polls = 0;
  const uint64_t t0 = ptx::globaltimer();
  for (;;) {
    ld_acquire_sys_v2(e, lo, hi);
    if ((uint32_t)lo == h + 1u && (uint32_t)(hi >> 32) == h + 1u) break;
    if ((++polls & 15u) == 0) {
      if (host_shutdown(a)) return false;
      if (ptx::globaltimer() - t0 > a.timeout_ns * 16 * a.lanes) {
        // the bound of one entry's wait, for each of the batch that a lane may wait behind
        record_status(a.status, GSYNC_ETIMEDOUT);
        return false;
      }
    }
  }
  const uint32_t req_len = (uint32_t)(lo >> 32), req_off = (uint32_t)hi, req_id = h;
  if (a.trace) a.trace[4ull * req_id] = ptx::globaltimer();
  const uint32_t s = claim_slot(a, h);
  if (s == kNoSlot) {
    record_status(a.status, GSYNC_ETIMEDOUT);
    return false;
  }
  Slot* sl = &a.slots[s];
  // Workers look at the claim word (and over-claims add to it) at any time, but read the rest only
  // after a claim of this request: everything is in place before the word is published.  An
  // over-claim of the slot's last request that lands before the publication is overwritten by it,
  // as one after it is a chunk of this request.
  const uint32_t nch = (req_len + a.chunk_elems - 1u) / a.chunk_elems;
  sl->id = req_id;
  sl->off = (int64_t)req_off;
  sl->len = (int64_t)req_len;
  sl->acc = 0ull;
  sl->done_chunks = 0u;
  ptx::st_release_u64(&sl->claim, (uint64_t)(nch == 0 ? 1u : nch) << 32);
  for (uint32_t m = 0; m < kMaskCopies; ++m) atomicOr(&a.active_mask[32u * m + (s >> 5)], 1u << (s & 31));
  ptx::red_add_relaxed(a.stats, 1u);
  if (a.trace) a.trace[4ull * req_id + 1] = ptx::globaltimer();
  return true;
}

// Three blocks per SM: the largest grid the registers have always allowed.
__global__ void __launch_bounds__(kThreads, 3) serve_kernel(Args a) {
  const uint32_t tid = threadIdx.x;
  const gsync::MutexRef lock = gsync::mutex_attach(a.ring_lock);
  const gsync::SemRef sem = gsync::sem_attach(a.admit_sem);
  __shared__ int s_cmd;             // 0 work, 1 exit, 2 nothing yet
  __shared__ int64_t s_lo[2], s_hi[2];  // the chunk to sum, and the next one (lo = hi: no more)
  const bool admitter = blockIdx.x < a.admitters;
  uint32_t idle = 0;
  uint64_t idle_since = 0;

  if (admitter) {
    // Admitters: ring indices (ticket lock) -> permits -> wait for those entries -> slots.
    // The indices and the permits are taken before the requests exist, so an arrival only
    // waits for one read of host memory.  A block admits `lanes` requests at a time, lane w
    // (thread 0 of warp w) the w-th of them.  What bounds a backlog is the ring lock's chain of
    // hand-offs: with one acquisition per request it took 0.83 us a request whatever the number
    // of admitters or the sizes; now one acquisition hands out a batch of indices.
    __shared__ uint32_t s_head;
    __shared__ int s_taken, s_left;  // written before one barrier each, and not again before the next
    const uint32_t lane = tid >> 5;
    if (lane >= a.lanes) return;
    if (tid == 0) s_left = 0;
    for (;;) {
      if (tid == 0) s_taken = take_indices(a, lock, s_head) ? 1 : 0;
      lanes_sync(a.lanes);
      if (!s_taken) return;
      if ((tid & 31u) == 0u && !admit(a, sem, s_head + lane)) s_left = 1;
      lanes_sync(a.lanes);
      if (s_left) return;
    }
  }

  // Workers: claim chunks of active slots until shutdown.  Thread 0 keeps the request's slot,
  // chunk count and value range.
  uint32_t seek = blockIdx.x * 0x85EBCA6Bu, slot = 0;
  Slot* sl = nullptr;
  uint32_t nchunks = 0, chunk = 0;
  bool backlog = false;
  int64_t off = 0, end = 0;
  auto set_chunk = [&](uint32_t c, uint32_t k) {
    const int64_t lo = off + (int64_t)c * a.chunk_elems;
    s_lo[k] = lo;
    s_hi[k] = lo + a.chunk_elems < end ? lo + a.chunk_elems : end;
  };
  for (;;) {
    if (tid == 0) {
      s_cmd = 2;  // nothing yet
      const uint32_t* my_mask = a.active_mask + 32u * (blockIdx.x % kMaskCopies);
      uint64_t mask;  // both mask words in one load (the copy starts a line)
      asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(mask) : "l"(my_mask) : "memory");
      // Visit only the set bits, from a place that differs from block to block and from look to
      // look, so that the workers spread over the active slots (all of them going on from the
      // slot they last served, they met at the next set bit and left most slots waiting).
      seek += 0x9E3779B1u;
      const uint32_t from = seek >> 26;
      const uint64_t upper = mask & (~0ull << from), lower = mask & ~(~0ull << from);
      bool got = false;
      for (int pass = 0; pass < 2 && !got; ++pass) {
        for (uint64_t m = pass ? lower : upper; m && !got; m &= m - 1u) {
          const uint32_t s = (uint32_t)__ffsll((long long)m) - 1u;
          if (!claim_chunk(&a.slots[s], chunk, nchunks)) continue;
          if (chunk + 1u == nchunks) retire_slot(a, s);
          sl = &a.slots[s];
          off = sl->off;
          end = off + sl->len;
          set_chunk(chunk, 0);
          if (a.trace && chunk == 0) a.trace[4ull * sl->id + 2] = ptx::globaltimer();
          s_cmd = 0;
          slot = s;
          backlog = __popcll((long long)mask) >= kBacklog;
          got = true;
        }
      }
      if (s_cmd == 2) {
        if ((idle & 15u) == 15u && ptx::ld_relaxed(a.dev_shutdown)) s_cmd = 1;
        if ((++idle & 255u) == 0) {
          if (ld_acquire_sys(a.shutdown)) s_cmd = 1;
          const uint64_t now = ptx::globaltimer();
          if (idle_since == 0) idle_since = now;
          else if (now - idle_since > a.timeout_ns * 16) { record_status(a.status, GSYNC_ETIMEDOUT); s_cmd = 1; }
        }
        if (s_cmd == 2) __nanosleep(32);
      } else {
        idle = 0;
        idle_since = 0;
      }
    }
    __syncthreads();
    const int cmd = s_cmd;
    if (cmd == 1) break;
    if (cmd == 2) { __syncthreads(); continue; }
    // With a backlog, up to kKeep chunks of this request in a row, added up in registers:
    // one reduction and one count of done chunks per block and request (with few requests in
    // flight other blocks are free, and a chunk taken early would only wait here).  Thread 0 asks
    // for the next one before it sums its share of this one, so the claim's round trip passes
    // under the loads.
    // No other request can take the slot meanwhile (this block's chunks are not counted done),
    // so the claim needs no look at the slot, and a claim past the last chunk ends it.
    long long sum = 0;
    uint32_t taken = 0;
    for (uint32_t k = 0;; k ^= 1u) {
      uint32_t next = nchunks;
      if (tid == 0 && backlog && taken + 1u < kKeep && chunk + 1u < nchunks)
        next = (uint32_t)ptx::atom_add_relaxed_u64(&sl->claim, 1ull);
      sum += thread_sum(a.pool, s_lo[k], s_hi[k]);
      ++taken;
      if (tid == 0) {
        chunk = next;
        if (chunk + 1u == nchunks) retire_slot(a, slot);
        if (chunk < nchunks) set_chunk(chunk, k ^ 1u);
        else s_lo[k ^ 1u] = s_hi[k ^ 1u] = 0;
      }
      __syncthreads();
      if (s_lo[k ^ 1u] == s_hi[k ^ 1u]) break;
    }
    const long long part = block_reduce(sum);
    if (tid == 0) {
      ptx::red_add_relaxed(a.stats + 32, taken);
      long long total = part;
      bool finished = taken == nchunks;  // the whole request: nothing to add up with other blocks
      if (!finished) {
        atomicAdd(&sl->acc, (unsigned long long)part);
        finished = ptx::atom_add_acq_rel(&sl->done_chunks, taken) + taken == nchunks;
        if (finished) total = (long long)ptx::ld_relaxed_u64((const uint64_t*)&sl->acc);
      }
      if (finished) {
        const uint32_t id = sl->id;
        if (a.trace) a.trace[4ull * id + 3] = ptx::globaltimer();
        st_relaxed_sys_s64(a.res + id, total);
        // One fence for everything this block hands on: the result and its flag to the host, the
        // slot to the next request, the permit to an admitter.  The stores after it have no order
        // among themselves, so none of them may touch the slot: its claim word, past the last
        // chunk, tells a worker that there is nothing left.
        asm volatile("fence.acq_rel.sys;" ::: "memory");
        st_relaxed_sys(a.done + id, 1u);
        free_slot(a, slot);
        ptx::red_add_relaxed(sem.word(2), 1u);  // the ticket window's post
        ptx::red_add_relaxed(a.stats + 64, 1u);
      }
    }
    __syncthreads();
  }
}

// Baseline: one launch per request; block j sums chunk j; the last block completes it.
__global__ void __launch_bounds__(kThreads) segsum_kernel(const int32_t* pool, int64_t off, int64_t len,
                                                          uint32_t chunk_elems, unsigned long long* acc,
                                                          uint32_t* counter, uint32_t id, int64_t* res,
                                                          uint32_t* done) {
  const int64_t lo = off + (int64_t)blockIdx.x * chunk_elems;
  int64_t hi = lo + chunk_elems;
  if (hi > off + len) hi = off + len;
  const long long part = block_reduce(thread_sum(pool, lo, hi));
  if (threadIdx.x == 0) {
    atomicAdd(acc, (unsigned long long)part);
    const uint32_t d = ptx::atom_add_acq_rel(counter, 1u) + 1u;
    if (d == gridDim.x) {
      const long long total = (long long)atomicAdd(acc, 0ull);
      st_relaxed_sys_s64(res + id, total);
      st_release_sys(done + id, 1u);
    }
  }
}

int host_dev_ptr(void* host, void** dev) {
  GSYNC_CUDA(cudaHostGetDevicePointer(dev, host, 0));
  return GSYNC_OK;
}

// The ring's device view.  Pinned host memory is mapped (host_dev_ptr).  A ring in managed
// memory has one address on both sides; on a GPU whose host reaches managed memory in place
// over a coherent link (cudaDevAttrDirectManagedMemAccessFromHost), it is advised to live in
// device memory and to stay mapped for the host, and is moved there before the host clears it:
// the producer's stores then cross the link into device memory, and the admitters poll it
// through the GPU's L2 instead of across the link.
int ring_device_ptr(void* ring, size_t bytes, cudaStream_t st, void** dev) {
  cudaPointerAttributes attr;
  GSYNC_CUDA(cudaPointerGetAttributes(&attr, ring));
  if (attr.type != cudaMemoryTypeManaged) return host_dev_ptr(ring, dev);
  int devid = 0, direct = 0;
  GSYNC_CUDA(cudaGetDevice(&devid));
  GSYNC_CUDA(cudaDeviceGetAttribute(&direct, cudaDevAttrDirectManagedMemAccessFromHost, devid));
  if (direct) {
    cudaMemLocation gpu = {};
    gpu.type = cudaMemLocationTypeDevice;
    gpu.id = devid;
    cudaMemLocation cpu = {};
    cpu.type = cudaMemLocationTypeHost;
    GSYNC_CUDA(cudaMemAdvise(ring, bytes, cudaMemAdviseSetPreferredLocation, gpu));
    GSYNC_CUDA(cudaMemAdvise(ring, bytes, cudaMemAdviseSetAccessedBy, cpu));
    GSYNC_CUDA(cudaMemPrefetchAsync(ring, bytes, gpu, 0, st));
    GSYNC_CUDA(cudaStreamSynchronize(st));
  }
  *dev = ring;
  return GSYNC_OK;
}

using Clock = std::chrono::steady_clock;

// Pins a host thread to one core (counted from the last core down) so that the producer and
// the collector are not descheduled behind each other.  Best effort: ignored on failure.
void pin_to_core_from_end(std::thread& t, int k) {
  const long n = sysconf(_SC_NPROCESSORS_ONLN);
  if (n < 4) return;
  cpu_set_t set;
  CPU_ZERO(&set);
  CPU_SET((int)(n - 1 - k), &set);
  (void)pthread_setaffinity_np(t.native_handle(), sizeof(set), &set);
}

int64_t now_ns(Clock::time_point t0) {
  return std::chrono::duration_cast<std::chrono::nanoseconds>(Clock::now() - t0).count();
}

void spin_until(Clock::time_point t) {
  while (Clock::now() < t) {
  }
}

// Counters shared by the host threads of a run, one per cache line: the collector updates
// `completed` (how many requests) and `prefix` (how many of the first, without a gap), which
// the calling thread and the producer read while the producer (or launcher) writes `published`, and
// a line shared between writers on different cores would bounce on every update.
struct alignas(128) HostCounter {
  std::atomic<int> v{0};
};
struct alignas(128) HostFlag {
  std::atomic<bool> v{false};
};

// Polls completion flags in order of arrival; records the host time each flag is first seen.
// A pass scans from the oldest incomplete request to the last one published (or launched), at
// most 4096 of them: only requests in flight can complete, so a pass stays as short as the
// work in flight instead of walking a fixed window of flags.
void collect(const gsync_serve_cfg* cfg, volatile uint32_t* done, Clock::time_point t0, const int64_t* sched,
             int64_t* lat, std::atomic<int>* completed, std::atomic<int>* prefix, std::atomic<bool>* abort_flag,
             const std::atomic<int>* published) {
  const int n = cfg->nreq;
  std::vector<char> seen(n, 0);
  int low = 0, count = 0, reported = 0, reported_low = 0;
  while (count < n && !abort_flag->load(std::memory_order_relaxed)) {
    const int hi = std::min(std::min(n, low + 4096), published->load(std::memory_order_acquire));
    for (int q = low; q < hi; ++q) {
      if (seen[q]) continue;
      if (done[q]) {
        std::atomic_thread_fence(std::memory_order_acquire);
        lat[q] = now_ns(t0) - sched[q];
        seen[q] = 1;
        ++count;
      }
    }
    while (low < n && seen[low]) ++low;
    if (low != reported_low) {
      prefix->store(low, std::memory_order_release);
      reported_low = low;
    }
    if (count != reported) {  // stored only when it moves, so readers keep the line cached
      completed->store(count, std::memory_order_release);
      reported = count;
    }
  }
}

// Every request must lie inside the pool and fit the chunk counter.
int check_requests(const gsync_serve_cfg* cfg, const gsync_serve_buffers* buf) {
  for (int q = 0; q < cfg->nreq; ++q) {
    const int64_t o = buf->offset[q], n = buf->length[q];
    if (o < 0 || n < 1 || o > buf->pool_elems - n) return GSYNC_EINVAL;
    if ((n + cfg->chunk_elems - 1) / cfg->chunk_elems > 32767) return GSYNC_EINVAL;
    if (q > 0 && buf->sched_ns[q] < buf->sched_ns[q - 1]) return GSYNC_EINVAL;
  }
  return GSYNC_OK;
}

// As many lanes as the permits cover with every admitter waiting for a full batch, up to one per
// warp; one lane where there are fewer slots than admitters.
uint32_t admission_lanes(const gsync_serve_cfg* cfg) {
  return (uint32_t)std::max(1, std::min(kThreads / 32, cfg->nslots / cfg->admitters));
}

}  // namespace

extern "C" size_t gsync_serve_workspace_bytes(int nslots) {
  if (nslots < 1 || nslots > 64) return 0;
  return 3 * 128 /* ring lock */ + 4 * 128 /* semaphore */ + (size_t)nslots * 128 +
         128 * kMaskCopies /* active mask */ + 3 * 128 /* stats */ + 128 /* status */ + 128 /* device shutdown */;
}

extern "C" int gsync_serve_run(const gsync_serve_cfg* cfg, gsync_serve_buffers* buf, void* workspace,
                               size_t workspace_bytes, void* stream) {
  if (!cfg || !buf || !workspace || cfg->nreq < 1 || cfg->nslots < 1 || cfg->nslots > 64 || cfg->nblocks < 2 ||
      cfg->admitters < 1 || cfg->admitters >= cfg->nblocks || cfg->chunk_elems < 1024 || cfg->ring_slots < 2 ||
      (cfg->ring_slots & (cfg->ring_slots - 1)) || !aligned(workspace, 256))
    return GSYNC_EINVAL;
  if (workspace_bytes < gsync_serve_workspace_bytes(cfg->nslots)) return GSYNC_EINVAL;
  if (!buf->pool || !buf->offset || !buf->length || !buf->sched_ns || !buf->ring || !buf->ctrl || !buf->res ||
      !buf->done || !buf->latency_ns)
    return GSYNC_EINVAL;
  if (int rc = check_requests(cfg, buf)) return rc;
  if (buf->pool_elems > (int64_t)0xFFFFFFFFll) return GSYNC_EINVAL;  // 32-bit offsets in the ring
  cudaStream_t st = (cudaStream_t)stream;
  char* p = (char*)workspace;
  uint32_t* ring_lock = (uint32_t*)p; p += 3 * 128;
  uint32_t* sem = (uint32_t*)p;       p += 4 * 128;
  Slot* slots = (Slot*)p;             p += (size_t)cfg->nslots * 128;
  uint32_t* mask = (uint32_t*)p;      p += 128 * kMaskCopies;
  uint32_t* stats = (uint32_t*)p;     p += 3 * 128;
  uint32_t* status = (uint32_t*)p;    p += 128;
  uint32_t* dev_shutdown = (uint32_t*)p;
  GSYNC_CUDA(cudaMemsetAsync(workspace, 0, gsync_serve_workspace_bytes(cfg->nslots), st));
  // Admitters may legitimately wait for a permit while arrivals are sparse (more admitters than
  // slots): the lock and the semaphore get 16x the per-wait bound.
  const uint64_t wait_ns = (cfg->timeout_ns ? cfg->timeout_ns : 2000000000ull) * 16;
  if (int rc = gsync_mutex_init(ring_lock, 3 * 128, GSYNC_MUTEX_TICKET, 1, nullptr, wait_ns, stream)) return rc;
  gsync_backoff sbo = {GSYNC_BACKOFF_EXPONENTIAL, 64, 2000, 0};
  if (int rc = gsync_sem_init(sem, 4 * 128, GSYNC_SEM_WINDOW, cfg->nslots, &sbo, wait_ns, stream)) return rc;

  // The host threads write these arrays on the latency path: touch every page first.
  for (int q = 0; q < cfg->nreq; ++q) buf->latency_ns[q] = 0;
  if (buf->publish_ns)
    for (int q = 0; q < cfg->nreq; ++q) buf->publish_ns[q] = 0;
  // Host control word ctrl[32] = shutdown; the ring starts empty (no entry has a valid seq).
  void* d_ring = nullptr;
  if (int rc = ring_device_ptr(buf->ring, kRingStride * (size_t)cfg->ring_slots, st, &d_ring)) return rc;
  volatile uint32_t* ctrl = buf->ctrl;
  ctrl[32] = 0;
  // Cleared as far as an admitter may look: the requests, and the batch that each admitter has
  // taken past them.  (All of a 65,536-entry ring is 8 MB, 90 us of a call.)
  const uint32_t lanes = admission_lanes(cfg);
  const int64_t polled = (int64_t)cfg->nreq + (int64_t)cfg->admitters * lanes;
  memset(buf->ring, 0, kRingStride * (size_t)std::min<int64_t>(cfg->ring_slots, polled));
  for (int q = 0; q < cfg->nreq; ++q) buf->done[q] = 0;
  std::atomic_thread_fence(std::memory_order_seq_cst);

  Args a;
  void *d_ctrl, *d_res, *d_done;
  if (int rc = host_dev_ptr((void*)buf->ctrl, &d_ctrl)) return rc;
  if (int rc = host_dev_ptr(buf->res, &d_res)) return rc;
  if (int rc = host_dev_ptr((void*)buf->done, &d_done)) return rc;
  a.ring = (const gsync_serve_req*)d_ring;
  a.ring_mask = (uint32_t)cfg->ring_slots - 1u;
  a.shutdown = (const uint32_t*)d_ctrl + 32;
  a.dev_shutdown = dev_shutdown;
  a.res = (int64_t*)d_res;
  a.done = (uint32_t*)d_done;
  a.pool = buf->pool;
  a.ring_lock = ring_lock;
  a.admit_sem = sem;
  a.slots = slots;
  a.active_mask = mask;
  a.stats = stats;
  a.status = status;
  a.busy = (unsigned long long*)(status + 16);  // the status line's second half
  a.trace = (unsigned long long*)buf->trace;
  a.nslots = (uint32_t)cfg->nslots;
  a.admitters = (uint32_t)cfg->admitters;
  a.chunk_elems = (uint32_t)cfg->chunk_elems;
  a.lanes = lanes;
  a.timeout_ns = cfg->timeout_ns ? cfg->timeout_ns : 2000000000ull;
  if (int rc = launch_coresident(serve_kernel, cfg->nblocks, kThreads, 1, 0, st, a)) return rc;

  // The loop is running (or about to): publish requests on their schedule, collect completions.
  std::this_thread::sleep_for(std::chrono::microseconds(cfg->start_delay_us));
  const Clock::time_point t0 = Clock::now();
  HostCounter completed_c, prefix_c, published_c;
  HostFlag abort_f;
  std::atomic<int>& completed = completed_c.v;
  std::atomic<int>&prefix = prefix_c.v, &published = published_c.v;
  std::atomic<bool>& abort_flag = abort_f.v;
  std::thread collector(collect, cfg, buf->done, t0, buf->sched_ns, buf->latency_ns, &completed, &prefix_c.v,
                        &abort_flag, &published);
  pin_to_core_from_end(collector, 1);
  const auto deadline = Clock::now() + std::chrono::nanoseconds(buf->sched_ns[cfg->nreq - 1]) +
                        std::chrono::seconds(cfg->drain_timeout_s);
  // The producer runs on its own pinned core too; this thread only waits.
  std::atomic<int> prod_rc{GSYNC_OK};
  std::thread producer([&]() {
    // Publishes every request whose time has come in one batch.  Each entry is written with
    // two aligned 8-byte stores, {seq, len} and {off, seq_check}, and no fence: each store is
    // single-copy atomic, so an entry whose seq and seq_check both read q + 1 holds request
    // q's len and off whatever order the two stores became visible in (a reader that sees
    // one half of an older lap's entry finds that half's sequence number stale).  One
    // write per half, with nothing to wait for between them, keeps the producer on schedule
    // where its stores cross the host link into device memory.
    int q = 0;
    while (q < cfg->nreq) {
      spin_until(t0 + std::chrono::nanoseconds(buf->sched_ns[q]));
      // The ring entry of request i is reused only after request i - ring_slots and all before it
      // completed.  (Requests complete in any order: their number says nothing about one entry.)
      int low;
      while (q - (low = prefix.load(std::memory_order_acquire)) >= cfg->ring_slots) {
        if (Clock::now() > deadline || abort_flag.load(std::memory_order_relaxed)) {
          prod_rc.store(GSYNC_ETIMEDOUT);
          return;
        }
      }
      // ... of which the ring takes as many as it has room for.
      const int room = (int)std::min<int64_t>(cfg->nreq, (int64_t)low + cfg->ring_slots);
      const int64_t now = now_ns(t0);
      int qe = q + 1;
      while (qe < room && buf->sched_ns[qe] <= now && qe - q < 64) ++qe;
      for (int i = q; i < qe; ++i) {
        uint64_t* e = (uint64_t*)((char*)buf->ring + (size_t)(i & (cfg->ring_slots - 1)) * kRingStride);
        const uint64_t seq = (uint32_t)(i + 1);
        // little-endian layout of gsync_serve_req: seq | len << 32, then off | seq_check << 32
        __atomic_store_n(e, seq | ((uint64_t)(uint32_t)buf->length[i] << 32), __ATOMIC_RELAXED);
        __atomic_store_n(e + 1, (uint64_t)(uint32_t)buf->offset[i] | (seq << 32), __ATOMIC_RELAXED);
      }
      published.store(qe, std::memory_order_release);
      if (buf->publish_ns) {
        const int64_t t = now_ns(t0);
        for (int i = q; i < qe; ++i) buf->publish_ns[i] = t;
      }
      q = qe;
    }
  });
  pin_to_core_from_end(producer, 0);
  int rc = GSYNC_OK;
  while (completed.load(std::memory_order_acquire) < cfg->nreq) {
    if (Clock::now() > deadline || prod_rc.load() != GSYNC_OK) {
      rc = GSYNC_ETIMEDOUT;
      break;
    }
    std::this_thread::sleep_for(std::chrono::microseconds(20));
  }
  abort_flag.store(true);
  producer.join();
  if (rc == GSYNC_OK) rc = prod_rc.load();
  collector.join();
  __atomic_store_n(&buf->ctrl[32], 1u, __ATOMIC_RELEASE);
  GSYNC_CUDA(cudaStreamSynchronize(st));
  uint32_t hstat[4 * 32];  // the three counters' lines and the status line, which follows them
  GSYNC_CUDA(cudaMemcpy(hstat, stats, sizeof hstat, cudaMemcpyDeviceToHost));
  for (int i = 0; i < 4; ++i) buf->stats[i] = hstat[32 * i];
  if (rc == GSYNC_OK && hstat[3 * 32]) rc = GSYNC_ETIMEDOUT;
  return rc;
}

extern "C" size_t gsync_serve_baseline_workspace_bytes(int nreq) {
  if (nreq < 1) return 0;
  return (size_t)nreq * 16;
}

extern "C" int gsync_serve_baseline(const gsync_serve_cfg* cfg, gsync_serve_buffers* buf, void* workspace,
                                    size_t workspace_bytes, void* const* streams, int nstreams) {
  if (!cfg || !buf || !workspace || cfg->nreq < 1 || cfg->chunk_elems < 1024 || !streams || nstreams < 1 ||
      workspace_bytes < gsync_serve_baseline_workspace_bytes(cfg->nreq) || !aligned(workspace, 16))
    return GSYNC_EINVAL;
  if (!buf->pool || !buf->offset || !buf->length || !buf->sched_ns || !buf->res || !buf->done || !buf->latency_ns)
    return GSYNC_EINVAL;
  if (int rc = check_requests(cfg, buf)) return rc;
  unsigned long long* acc = (unsigned long long*)workspace;
  uint32_t* counter = (uint32_t*)(acc + cfg->nreq);
  GSYNC_CUDA(cudaMemsetAsync(workspace, 0, gsync_serve_baseline_workspace_bytes(cfg->nreq), (cudaStream_t)streams[0]));
  GSYNC_CUDA(cudaStreamSynchronize((cudaStream_t)streams[0]));
  for (int q = 0; q < cfg->nreq; ++q) buf->done[q] = 0;
  for (int q = 0; q < cfg->nreq; ++q) buf->latency_ns[q] = 0;
  if (buf->publish_ns)
    for (int q = 0; q < cfg->nreq; ++q) buf->publish_ns[q] = 0;
  std::atomic_thread_fence(std::memory_order_seq_cst);
  void *d_res, *d_done;
  if (int rc = host_dev_ptr(buf->res, &d_res)) return rc;
  if (int rc = host_dev_ptr((void*)buf->done, &d_done)) return rc;
  const Clock::time_point t0 = Clock::now();
  HostCounter completed_c, prefix_c, published_c;
  HostFlag abort_f;
  std::atomic<int>& completed = completed_c.v;
  std::atomic<int>& published = published_c.v;
  std::atomic<bool>& abort_flag = abort_f.v;
  std::thread collector(collect, cfg, buf->done, t0, buf->sched_ns, buf->latency_ns, &completed, &prefix_c.v,
                        &abort_flag, &published);
  pin_to_core_from_end(collector, 1);
  int dev = 0;
  GSYNC_CUDA(cudaGetDevice(&dev));
  std::atomic<int> launch_rc{GSYNC_OK};
  // The launching loop runs on its own pinned core, like the persistent loop's producer.
  std::thread launcher([&]() {
    if (cudaSetDevice(dev) != cudaSuccess) {
      launch_rc.store(GSYNC_ECUDA);
      return;
    }
    for (int q = 0; q < cfg->nreq; ++q) {
      spin_until(t0 + std::chrono::nanoseconds(buf->sched_ns[q]));
      const int64_t len = buf->length[q];
      const unsigned nb = (unsigned)((len + cfg->chunk_elems - 1) / cfg->chunk_elems);
      segsum_kernel<<<nb, kThreads, 0, (cudaStream_t)streams[q % nstreams]>>>(
          buf->pool, buf->offset[q], len, (uint32_t)cfg->chunk_elems, acc + q, counter + 2 * q, (uint32_t)q,
          (int64_t*)d_res, (uint32_t*)d_done);
      // The collector's scan bound, 16 launches ahead, moved once every 16 launches: a store
      // per launch would bounce the line between this core and the collector's, and this
      // loop is what limits the arm at high rates.
      if ((q & 15) == 0) published.store(std::min(cfg->nreq, q + 16), std::memory_order_release);
      if (buf->publish_ns) buf->publish_ns[q] = now_ns(t0);
      if (cudaGetLastError() != cudaSuccess) {
        launch_rc.store(GSYNC_ECUDA);
        return;
      }
    }
  });
  pin_to_core_from_end(launcher, 0);
  launcher.join();
  int rc = launch_rc.load();
  const auto deadline = Clock::now() + std::chrono::seconds(cfg->drain_timeout_s);
  while (rc == GSYNC_OK && completed.load(std::memory_order_acquire) < cfg->nreq) {
    if (Clock::now() > deadline) rc = GSYNC_ETIMEDOUT;
    std::this_thread::sleep_for(std::chrono::microseconds(20));
  }
  abort_flag.store(true);
  collector.join();
  for (int s = 0; s < nstreams; ++s) GSYNC_CUDA(cudaStreamSynchronize((cudaStream_t)streams[s]));
  return rc;
}

namespace {

__global__ void host_pingpong_kernel(uint32_t* words, int iters, uint32_t* status) {
  // words[0]: device -> host, words[32]: host -> device (separate lines).
  const uint64_t deadline = ptx::globaltimer() + 2000000000ull;
  for (int i = 1; i <= iters; ++i) {
    st_release_sys(words, (uint32_t)i);
    uint32_t polls = 0;
    while (ld_acquire_sys(words + 32) != (uint32_t)i) {
      if ((++polls & 63u) == 0 && ptx::globaltimer() > deadline) {
        *status = 1;
        st_release_sys(words, 0xFFFFFFFFu);  // tells the host thread to stop
        return;
      }
    }
  }
}

}  // namespace

extern "C" int gsync_probe_host_pingpong(uint32_t* words, int iters, uint64_t* out_ns, void* stream) {
  if (!words || !out_ns || iters < 1) return GSYNC_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  void* dwords = nullptr;
  if (int rc = host_dev_ptr(words, &dwords)) return rc;
  volatile uint32_t* w = words;
  w[0] = 0;
  w[32] = 0;
  w[48] = 0;  // device-side status word
  std::atomic_thread_fence(std::memory_order_seq_cst);
  host_pingpong_kernel<<<1, 1, 0, st>>>((uint32_t*)dwords, iters, (uint32_t*)dwords + 48);
  GSYNC_CUDA(cudaGetLastError());
  const auto deadline = Clock::now() + std::chrono::seconds(5);
  Clock::time_point t0 = Clock::now();
  bool ok = true;
  for (int i = 1; i <= iters && ok; ++i) {
    uint32_t v;
    while ((v = __atomic_load_n(&words[0], __ATOMIC_ACQUIRE)) != (uint32_t)i) {
      if (v == 0xFFFFFFFFu || Clock::now() > deadline) { ok = false; break; }
    }
    if (i == 1) t0 = Clock::now();
    __atomic_store_n(&words[32], (uint32_t)i, __ATOMIC_RELEASE);
  }
  const auto t1 = Clock::now();
  GSYNC_CUDA(cudaStreamSynchronize(st));
  if (!ok || w[48]) return GSYNC_ETIMEDOUT;
  out_ns[0] = (uint64_t)std::chrono::duration_cast<std::chrono::nanoseconds>(t1 - t0).count();
  return GSYNC_OK;
}
