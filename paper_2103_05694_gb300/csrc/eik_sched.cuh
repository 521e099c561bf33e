// Device helpers and the bucket scheduler shared by the tile kernels
// (eik_solver.cu, eik_front.cu, eik_guided.cu, eik_adjoint.cu): bit-pattern arithmetic, relaxed and
// acquire/release accesses, and the ring of bucket slots (push, pop, claim,
// finish).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "eik_exact.cuh"
#include "eik_internal.h"

// The functions of the scheduler proper (left to the compiler unless a file asks).
#ifndef EIK_SCHED_FN
#define EIK_SCHED_FN __device__
#endif

// Whether a wait for work looks at SolveParams::progress before it gives up (only where
// a file asks: in the guided kernel, bound by instruction fetch, the branch costs 0.3 %).
#ifndef EIK_SCHED_PROGRESS
#define EIK_SCHED_PROGRESS 0
#endif

namespace eik {
namespace {

constexpr unsigned long long kInfBits = 0x7ff0000000000000ull;
constexpr unsigned kFull = 0xffffffffu;
constexpr unsigned kMaxRounds = 1u << 20;   // per tile visit; never reached in practice

__device__ __forceinline__ unsigned long long bits_of(double x) {
  return static_cast<unsigned long long>(__double_as_longlong(x));
}
__device__ __forceinline__ double from_bits(unsigned long long u) {
  return __longlong_as_double(static_cast<long long>(u));
}
__device__ __forceinline__ unsigned long long umin64(unsigned long long a, unsigned long long b) {
  return a < b ? a : b;
}
__device__ __forceinline__ unsigned long long umax64(unsigned long long a, unsigned long long b) {
  return a < b ? b : a;
}

// Minimum of a 64-bit value over the full warp with two warp-reduce
// instructions (high words first, then the low words of the lanes that hold
// the smallest high word).
__device__ __forceinline__ unsigned long long warp_min64(unsigned long long v) {
  const unsigned hi = __reduce_min_sync(0xffffffffu, static_cast<unsigned>(v >> 32));
  const unsigned lo = __reduce_min_sync(
      0xffffffffu, static_cast<unsigned>(v >> 32) == hi ? static_cast<unsigned>(v) : 0xffffffffu);
  return (static_cast<unsigned long long>(hi) << 32) | lo;
}

// Phase timing (counters >= 2, thread 0): add the cycles since the last lap
// to slot k of the CTA's statistics (slot 12 holds the last lap's clock).
__device__ __forceinline__ void lap(long long *st, int k) {
  const long long c1 = clock64();
  st[k] += c1 - st[12];
  st[12] = c1;
}

// One axis of a cell after an acceptance step: sides (left/right) with their
// values after the step and whether they changed (decreased).  True when the
// axis minimum decreased and is now below `best`: the smallest changed value
// lies below every unchanged side's value and below `best`.
__device__ __forceinline__ bool axis_fell(bool c1, unsigned long long v1, bool c2,
                                          unsigned long long v2, unsigned long long best) {
  const unsigned long long lowered = umin64(c1 ? v1 : kInfBits, c2 ? v2 : kInfBits);
  const unsigned long long kept = umin64(c1 ? kInfBits : v1, c2 ? kInfBits : v2);
  return lowered < kept && lowered < best;
}

// A cell's candidate is pending while it differs from the cell's value
// (+inf: none); accepting it sets the value to it.
__device__ __forceinline__ bool is_pending(unsigned long long pv, unsigned long long t) {
  return pv != t && pv != kInfBits;
}

// Orders this thread's earlier accesses before its later ones for threads that
// synchronise with it (cheaper than __threadfence(), which is sequentially
// consistent).
__device__ __forceinline__ void fence_ar() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// Relaxed, GPU-scope accesses (never served from a stale L1 line).
__device__ __forceinline__ unsigned ld_rlx(const unsigned *p) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ int ld_rlx(const int *p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long ld_rlx(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ double ld_time(const double *p) {
  double v;
  asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_rlx(unsigned long long *p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void st_rlx(unsigned *p, unsigned v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// Atomics that publish (release) or take over (acquire) a ring entry.
__device__ __forceinline__ unsigned long long cas_rel(unsigned long long *p, unsigned long long old,
                                                      unsigned long long v) {
  unsigned long long r;
  asm volatile("atom.release.gpu.global.cas.b64 %0, [%1], %2, %3;" : "=l"(r) : "l"(p), "l"(old), "l"(v) : "memory");
  return r;
}
__device__ __forceinline__ unsigned long long exch_acq(unsigned long long *p, unsigned long long v) {
  unsigned long long r;
  asm volatile("atom.acquire.gpu.global.exch.b64 %0, [%1], %2;" : "=l"(r) : "l"(p), "l"(v) : "memory");
  return r;
}
__device__ __forceinline__ long long now_ns() {
  long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ void raise_status(Ctl *ctl, unsigned code, unsigned long long info) {
  if (atomicCAS(&ctl->status, 0u, code) == 0u) {
    ctl->error_info[0] = info;
  }
}

// ---------------------------------------------------------------------------
// Scheduler.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long make_state(unsigned long long st, unsigned bucket,
                                                         unsigned faces) {
  return (st << 40) | (static_cast<unsigned long long>(faces) << 32) | bucket;
}
__device__ __forceinline__ unsigned long long state_of(unsigned long long s) { return (s >> 40) & 3ull; }
__device__ __forceinline__ unsigned bucket_of(unsigned long long s) {
  return static_cast<unsigned>(s & 0x3fffffffull);
}
__device__ __forceinline__ unsigned faces_of(unsigned long long s) {
  return static_cast<unsigned>((s >> 32) & 0x7full);
}

__device__ __forceinline__ unsigned bucket_of_time(unsigned long long tb, float inv_delta) {
  const float q = xf::to_f(tb) * inv_delta;   // no FP64-pipe conversion
  if (!(q < static_cast<float>(kMaxBucket))) return kMaxBucket;
  return static_cast<unsigned>(q);
}

// Append (tile, b) to bucket b's slot.  The caller already owns the right to
// push (it moved the tile's state to queued(b)).
EIK_SCHED_FN bool push_entry(const SolveParams &p, unsigned long long tile, unsigned b) {
  Ctl *ctl = p.ctl;
  atomicAdd(&ctl->work, 1);
  const unsigned s = b & (kNumSlots - 1);
  const unsigned cap = p.cap_mask + 1u;
  const unsigned idx = atomicAdd(&ctl->push[s * kCounterPad], 1u);
  unsigned long long *const slot = p.slots + static_cast<size_t>(s) * cap + (idx & p.cap_mask);
  const unsigned long long e = (static_cast<unsigned long long>(b + 1u) << 32) | tile;
  long long t0 = 0;
#pragma unroll 1
  while (cas_rel(slot, 0ull, e) != 0ull) {   // the position still holds an entry of an earlier lap
    // depth as a signed difference: a popper may already have taken index idx
    if (static_cast<int>(idx - ld_rlx(&ctl->pop[s * kCounterPad])) >= static_cast<int>(cap)) {
      raise_status(ctl, kEcapacity, (static_cast<unsigned long long>(s) << 32) | idx);
      return false;
    }
    const long long now = now_ns();
    if (t0 == 0) t0 = now;
    else if (now - t0 > p.timeout_ns) { raise_status(ctl, kEcapacity, 1ull << 63); return false; }
    if (ld_rlx(&ctl->status)) return false;
    __nanosleep(64);
  }
  // the entry is written: one more for poppers to reserve
  atomicAdd(&ctl->avail[s * kCounterPad], 1);
  // A scanner may have moved the lowest-bucket hint past this slot between
  // the caller's read of the hint and the push: pull the hint back.  A
  // scanner's forward CAS from a stale value then fails.
  atomicMin(&ctl->cur, b);
  if (p.counters) {
    atomicAdd(&ctl->stats[kStatPushes], 1ull);
    const int depth = static_cast<int>(idx - ld_rlx(&ctl->pop[s * kCounterPad]));
    if (depth > 0) atomicMax(&ctl->stats[kStatMaxQueue], static_cast<unsigned long long>(depth));
  }
  return true;
}

// A face of `tile` has new lower halo values (the smallest in bucket
// `bucket`): make sure the tile is (re)processed after this point.  cur: the
// lowest-bucket hint, now or a little earlier (it only clamps the priority).
EIK_SCHED_FN void activate(const SolveParams &p, unsigned long long tile, unsigned face_bits,
                           unsigned bucket, unsigned cur) {
  Ctl *ctl = p.ctl;
  unsigned b = bucket;
  if (b < cur) b = cur;
  else if (b - cur >= kNumSlots) b = cur + kNumSlots - 1;
  if (b > kMaxBucket) b = kMaxBucket;
  unsigned long long old = 0ull;          // idle, most often; the CAS tells otherwise
#pragma unroll 1
  for (int it = 0; it < (1 << 22); ++it) {
    const unsigned long long st = state_of(old);
    const unsigned ob = bucket_of(old), of = faces_of(old);
    unsigned long long nw;
    bool need_push = false;
    if (st == kStIdle) {
      nw = make_state(kStQueued, b, face_bits);
      need_push = true;
    } else if (st == kStQueued) {
      nw = make_state(kStQueued, b < ob ? b : ob, of | face_bits);
      need_push = b < ob;
    } else if (st == kStRunning) {
      nw = make_state(kStDirty, b, face_bits);
    } else {
      nw = make_state(kStDirty, b < ob ? b : ob, of | face_bits);
    }
    if (nw == old) return;
    const unsigned long long prev = atomicCAS(&p.state[tile], old, nw);
    if (prev == old) {
      if (need_push) push_entry(p, tile, b);
      return;
    }
    old = prev;
  }
  raise_status(ctl, kEtimeout, 3);
}

__device__ __forceinline__ void activate(const SolveParams &p, unsigned long long tile,
                                         unsigned face_bits, unsigned bucket) {
  activate(p, tile, face_bits, bucket, ld_rlx(&p.ctl->cur));
}

// Claim a popped entry: queued(b) -> running.  Returns the face mask, or -1
// if the entry is stale (the tile was re-queued elsewhere or is done).
EIK_SCHED_FN int try_claim(const SolveParams &p, unsigned long long tile, unsigned b) {
  unsigned long long old = ld_rlx(&p.state[tile]);
#pragma unroll 1
  for (int it = 0; it < (1 << 22); ++it) {
    if (state_of(old) != kStQueued || bucket_of(old) != b) return -1;
    const unsigned long long prev = atomicCAS(&p.state[tile], old, make_state(kStRunning, 0, 0));
    if (prev == old) return static_cast<int>(faces_of(old));
    old = prev;
  }
  raise_status(p.ctl, kEtimeout, 4);
  return -1;
}

// End of a visit: running -> idle, or dirty(b) -> queued(b) plus a push.
EIK_SCHED_FN void finish_tile(const SolveParams &p, unsigned long long tile) {
  unsigned long long old = make_state(kStRunning, 0, 0);
#pragma unroll 1
  for (int it = 0; it < (1 << 22); ++it) {
    unsigned long long nw;
    const bool dirty = state_of(old) == kStDirty;
    nw = dirty ? make_state(kStQueued, bucket_of(old), faces_of(old)) : 0ull;
    const unsigned long long prev = atomicCAS(&p.state[tile], old, nw);
    if (prev == old) {
      if (dirty) push_entry(p, tile, bucket_of(old));
      return;
    }
    old = prev;
  }
  raise_status(p.ctl, kEtimeout, 5);
}

// The same for the kernels that go on with a tile at once when it was re-activated
// meanwhile: running -> idle (returns 0), or dirty -> running (0x100 | the new
// faces).  One thread, after a barrier with the threads that stored the tile's
// cells.  The fence makes the state a release of all of these stores: the next
// visitor loads the cells with relaxed loads and stores over them, so a value that
// it missed would be lost.
__device__ __forceinline__ int end_visit(const SolveParams &p, unsigned long long tile) {
  fence_ar();
  const unsigned long long mine = make_state(kStRunning, 0, 0);
  unsigned long long old = mine;
#pragma unroll 1
  for (int it = 0; it < (1 << 22); ++it) {
    const unsigned long long prev = atomicCAS(&p.state[tile], old, old == mine ? 0ull : mine);
    if (prev == old) {
      if (old == mine) return 0;
      fence_ar();   // the claim of the new work before the halo loads
      return 0x100 | static_cast<int>(faces_of(old));
    }
    old = prev;
  }
  raise_status(p.ctl, kEtimeout, 5);
  return 0;
}

// The entry at index q of slot s (reserved by the caller), freeing its position:
// waits until a pusher has written it.  (If laps meet at a position, the
// entries go to either taker: they are all live.)
EIK_SCHED_FN unsigned long long take_slot(const SolveParams &p, unsigned s, unsigned q) {
  unsigned long long *const slot = p.slots + static_cast<size_t>(s) * (p.cap_mask + 1u) + (q & p.cap_mask);
  long long t0 = 0;
#pragma unroll 1
  for (;;) {
    const unsigned long long e = exch_acq(slot, 0ull);
    if (e != 0ull) return e - (1ull << 32);
    const long long now = now_ns();
    if (t0 == 0) t0 = now;
    else if (now - t0 > p.timeout_ns) { raise_status(p.ctl, kEtimeout, 6); return kEmpty; }
    if (ld_rlx(&p.ctl->status)) return kEmpty;
    __nanosleep(32);
  }
}

// Warp 0: take one entry from the lowest active bucket slots.  A slot is
// active while it holds entries or tiles claimed from it are still running;
// the hint `cur` moves up to the lowest active slot, and only slots within
// `window` buckets of it are popped (bounded look-ahead, the soft priority of
// OBIM).  On success the slot's run counter has been incremented for the
// caller, `slot_out` is the slot and `lo_out` the lowest active bucket.
// Returns kEmpty when the solve is over (done or error).  The wait gives up
// timeout_ns after the last entry taken (idle_since), or, with EIK_SCHED_PROGRESS, when
// the caller's count has stood still for so long.
EIK_SCHED_FN unsigned long long pop_entry(const SolveParams &p, long long &idle_since,
                                        unsigned &slot_out, unsigned &lo_out) {
  Ctl *ctl = p.ctl;
  const unsigned lane = threadIdx.x & 31u;
  const unsigned win = p.window < 31u ? p.window : 31u;
  unsigned nap = 64;
  unsigned long long seen = 0ull;       // *p.progress when idle_since was set
#pragma unroll 1
  for (;;) {
    unsigned stop = 0, cur = 0;
    if (lane == 0) {
      cur = ld_rlx(&ctl->cur);
      stop = ld_rlx(&ctl->status) | ld_rlx(&ctl->done);
    }
    stop = __shfl_sync(kFull, stop, 0);
    if (stop) return kEmpty;
    cur = __shfl_sync(kFull, cur, 0);
    // find the lowest active slot at or above the hint (whole ring if needed)
    unsigned first = 0xffffffffu;
    unsigned s = 0;
    bool pend = false;
#pragma unroll 1
    for (unsigned base = 0; base < kNumSlots; base += 32) {
      s = (cur + base + lane) & (kNumSlots - 1);
      const int av = ld_rlx(&ctl->avail[s * kCounterPad]);
      const unsigned rn = p.gate_pending_only ? 0u : ld_rlx(&ctl->run[s * kCounterPad]);
      pend = av > 0;
      const unsigned act = __ballot_sync(kFull, pend || rn > 0u);
      if (act) {
        first = base + static_cast<unsigned>(__ffs(act) - 1);
        break;
      }
    }
    if (first == 0xffffffffu) {
      int w = 0;
      if (lane == 0) w = ld_rlx(&ctl->work);
      w = __shfl_sync(kFull, w, 0);
      if (w == 0) {
        if (lane == 0) st_rlx(&ctl->done, 1u);
        return kEmpty;
      }
    } else {
      if (first > 0 && lane == 0 && cur + first <= kMaxBucket) atomicCAS(&ctl->cur, cur, cur + first);
      if (first >= 32) continue;   // re-read the 32 slots from the new hint
      const unsigned lo = cur + first;
      unsigned cand = __ballot_sync(kFull, pend && lane >= first && lane <= first + win);
#pragma unroll 1
      while (cand) {
        const int l = __ffs(cand) - 1;
        unsigned long long e = kEmpty;
        int got = 0;
        if (lane == static_cast<unsigned>(l)) {
          atomicAdd(&ctl->run[s * kCounterPad], 1u);   // keep the slot active meanwhile
          // reserve one written entry, then take the next index: two
          // fetch-and-adds, so many idle CTAs never serialise on a retried CAS.
          // Reservations never exceed the entries written, so pop <= push.  Only
          // a popper that has just seen an entry to reserve tries (a failed try
          // holds the count down until it is undone).
          int *av = &ctl->avail[s * kCounterPad];
          if (atomicAdd(av, -1) > 0) {
            got = 1;
            e = take_slot(p, s, atomicAdd(&ctl->pop[s * kCounterPad], 1u));
          } else {
            atomicAdd(av, 1);                           // nothing left: undo the try
          }
          if (!got) atomicAdd(&ctl->run[s * kCounterPad], 0xffffffffu);
        }
        got = __shfl_sync(kFull, got, l);
        if (got) {
          e = __shfl_sync(kFull, e, l);
          slot_out = __shfl_sync(kFull, s, l);
          lo_out = lo;
          return e;  // kEmpty here means the solve is being aborted
        }
        cand &= ~(1u << l);
      }
    }
    if (lane == 0) {
      const long long now = now_ns();
      if (idle_since == 0) {
        idle_since = now;
        if (EIK_SCHED_PROGRESS) seen = ld_rlx(p.progress);
      } else if (now - idle_since > p.timeout_ns) {
        const unsigned long long got = EIK_SCHED_PROGRESS ? ld_rlx(p.progress) : seen;
        if (got == seen) raise_status(ctl, kEtimeout, 2);
        seen = got;
        idle_since = now;
      }
    }
    // longer and longer: a scan is 66 L2 reads of lines that the working CTAs'
    // atomics need, and with many idle CTAs one looks soon anyway (24 sections of
    // 150 to 400 by 300 to 800 cells: 2.87 ms at a fixed 128 ns, 2.65 with this;
    // adjoints of one to four 600 x 500 fields, with CTAs by their size: the same)
    __nanosleep(nap);
    nap = nap < 4096u ? 2u * nap : 4096u;
  }
}

__device__ __forceinline__ int find_prob(const SolveParams &p, unsigned long long tile) {
  int lo = 0, hi = p.nprob - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (static_cast<unsigned long long>(p.probs[mid].tile_base) <= tile) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ bool is_source(const Prob &P, int64_t idx) {
  int64_t lo = 0, hi = P.nsrc - 1;
  while (lo <= hi) {
    const int64_t mid = (lo + hi) >> 1;
    const int64_t v = P.src_idx[mid];
    if (v == idx) return true;
    if (v < idx) lo = mid + 1; else hi = mid - 1;
  }
  return false;
}

// ---------------------------------------------------------------------------
// Shared by the kernels that give a tile to one warp.
// ---------------------------------------------------------------------------
// A 64-bit field of a record that no kernel writes, through the read-only path.
__device__ __forceinline__ int64_t ldg_i64(const void *p) {
  return __ldg(static_cast<const long long *>(p));
}

__device__ __forceinline__ int find_prob_ro(const SolveParams &p, unsigned tile) {
  int lo = 0, hi = p.nprob - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (ldg_i64(&p.probs[mid].tile_base) <= static_cast<int64_t>(tile)) lo = mid; else hi = mid - 1;
  }
  return lo;
}

constexpr float kInfF = __builtin_huge_valf();

// A non-negative double (bit pattern) times 2^-se as a float, truncated; +inf stays.
__device__ __forceinline__ float to_f_scaled(unsigned long long u, int se) {
  const int e = static_cast<int>(u >> 52) - 1023 + 127 - se;
  if (u == 0ull || e <= 0) return 0.0f;
  if (e >= 255) return kInfF;
  return __int_as_float((e << 23) | static_cast<int>((u >> 29) & 0x7fffffu));
}

// Bit sets over a tile's cells: lane k < NC holds the word of cells 32 k .. 32 k + 31
// (the other lanes 0).  For every cell q the bit of cell q + d; bits whose
// neighbour is off the tile mean nothing and are masked by the caller.
template <int d>
__device__ __forceinline__ unsigned nbr_bits(unsigned w, bool across) {
  constexpr int m = d < 0 ? -d : d;
  if (m >= 32) {
    if (d > 0) return __shfl_down_sync(kFull, w, m / 32);
    const unsigned v = __shfl_up_sync(kFull, w, m / 32);
    return (threadIdx.x & 31) >= m / 32 ? v : 0u;
  }
  unsigned r = d > 0 ? w >> m : w << m;
  if (across) {        // the neighbour may be in the next word
    if (d > 0) {
      r |= __shfl_down_sync(kFull, w, 1) << (32 - m);
    } else {
      const unsigned v = __shfl_up_sync(kFull, w, 1) >> (32 - m);
      r |= (threadIdx.x & 31) > 0 ? v : 0u;
    }
  }
  return r;
}

// The bits of the neighbours across face j (-x, +x, -y, +y, -z, +z) of the cells of
// a TX x TY x TZ tile, cells numbered x fastest.
template <int TX, int TY, int TZ>
__device__ __forceinline__ unsigned face_bits(unsigned w, int j) {
  switch (j) {
    case 0: return nbr_bits<-1>(w, false);
    case 1: return nbr_bits<1>(w, false);
    case 2: return nbr_bits<-TX>(w, TX * TY > 32);
    case 3: return nbr_bits<TX>(w, TX * TY > 32);
    case 4: return nbr_bits<-TX * TY>(w, true);
    default: return nbr_bits<TX * TY>(w, true);
  }
}

// A set's cells as a list in shared memory (to be read after a __syncwarp);
// returns their number.  Each word's lane writes its bits (every lane picking its
// bit of each word in turn: 29.0 against 14.7 kcycles a visit for 8 words).
template <int NC>
__device__ __forceinline__ int list_of_set(unsigned set, unsigned char *list) {
  const int lane = threadIdx.x & 31;
  const int own = __popc(set);
  int n = own;
#pragma unroll
  for (int o = 1; o < NC; o <<= 1) {
    const int v = __shfl_up_sync(kFull, n, o);
    if (lane >= o) n += v;
  }
  int at = n - own;
  n = __shfl_sync(kFull, n, NC - 1);
#pragma unroll 1
  for (unsigned w = set; w; w &= w - 1u) list[at++] = static_cast<unsigned char>(lane * 32 + __ffs(w) - 1);
  return n;
}

}  // namespace
}  // namespace eik
