// Front kernel: the tile kernel of lean solves with automatic options, except 3D
// batches that fill the device (eik_guided.cu).
//
// What bounds a solve with few fronts is the chain of cells along them: a cell can
// be final one evaluation after its upwind neighbours, so the kernel is built
// around a short step, and around tiles that advance together:
//  * A tile has 64 cells (8x8, 4x4x4) and a CTA of two warps: one cell per thread,
//    whose value, constant and masks stay in registers.  A round evaluates by d-bar
//    every cell with a neighbour that fell in the last round, publishes what fell
//    (one ballot word per warp) and meets at one barrier.  No order is kept: a
//    round costs the same for 1 or 64 cells, and a cell whose upwind cells are
//    final is final one round later whatever the others do.
//  * Halos are live: every value that falls is stored at once, and every round
//    reloads the halo (the load overlaps the evaluations), so neighbouring tiles
//    that are being visited exchange fronts cell by cell.  A tile is activated when
//    a first value below its halo value appears on its face, and once more at
//    the end of the visit if there were later ones.
// Reads and writes of one word by two threads in a round are harmless: a value
// only falls, is a valid upper bound at any time, and whoever may have missed a
// fall is evaluated again in the next round.  A visit ends after a round in which
// nothing fell, inside or on the halo, and no activation came meanwhile; the
// next visit evaluates every cell beside a finite halo value, since it cannot tell
// which of these its predecessor has seen.  So when no tile is active no
// evaluation would lower a value: the fixed point and its bits are those of any
// schedule (Theorem 1).
//
// Measured against the guided kernel (FP32 order, then one exact evaluation per
// cell; us for the solve): 129^2 grid 483 -> 250, 20 x 21 x 22 grid 800 -> 300,
// 751 x 2301 layered section 9264 -> 4086, 97 x 131 x 203 grid 3176 -> 1820, 256^3
// checkerboard 11082 -> 8030, 24 ragged sections 3510 -> 1916, 32 sources of
// 1024^2 13262 -> 11214; a layered section takes about 1950 cycles per cell of its
// longest chain.  It evaluates a cell more often (28 times on the section), so
// where there are fronts enough to fill the device with ordered work the guided
// kernel stays ahead (88-problem 3D batch: 43 against 78 ms).
// One warp of two cells per lane: 5290 against 4086 us on the section (1.7
// evaluations per round), but 7.6 against 8.0 ms on the checkerboard.
// In 2D, where CTAs are free for it (SolveParams::ahead), a tile that a first front
// reaches activates the neighbours that none has reached, and such a tile looks at
// its halo for up to 16 rounds: starting a visit (push, pop, claim, loads: about 12
// kcycles) then overlaps the front's way through the tile before (8 rounds of 1900;
// a strip of 8 x 4096 cells 7.4 -> 5.7 ms, 129^2 252 -> 217 us, the section 3900 ->
// 3180, 1502 x 4602 8980 -> 7360, 24 ragged sections 1724 -> 1520).  3D tiles are
// reached from several sides, and the waiting CTAs are missed: checkerboard 7.6 ->
// 8.6 ms, 97 x 131 x 203 1.68 -> 1.74; 32 sources of 1024^2 10.8 -> 11.3 ms.
// With few fronts a third warp activates the neighbours (an activation is a fence
// and three dependent atomics, 5 kcycles, about 1.5 times a visit), so that the rounds
// go on meanwhile: 129^2 219 -> 205 us, the section 3150 -> 3030, 1502 x 4602 7360 ->
// 6700.  It also claims the tiles and ends the visits; its mailbox takes the bucket
// time of each face.
// Waiting a few rounds before any visit ends: no gain (5.25 -> 5.3 ms).
#include <cstdint>
#include <cuda_runtime.h>

#include "eik_exact.cuh"
#include "eik_internal.h"
#define EIK_SCHED_FN __device__ __noinline__
#include "eik_sched.cuh"

namespace eik {
namespace {

// The third warp's part of a visit: deliver the mail (lane j < 4: the bucket time of
// face j) until the rounds are over (*fin) and no mail is left.  The rounds end
// by themselves, after kMaxRounds at the latest, whatever timeout_ms is, so the
// wait's own limit lies beyond that (a round takes about 1 us); lane 0 looks at the
// clock for the whole warp, since the lanes' clocks differ and the votes need all of them.
constexpr long long kVisitNs = 10ll * 1000 * 1000 * 1000;
template <class Deliver>
__device__ __forceinline__ void serve_mail(unsigned long long *mail, volatile int *fin, const SolveParams &p,
                                           Deliver deliver) {
  const int lane = threadIdx.x & 31;
  const long long limit = p.timeout_ns > kVisitNs ? p.timeout_ns : kVisitNs;
  long long t0 = 0;
#pragma unroll 1
  for (unsigned it = 0;; ++it) {
    const bool over = *fin != 0;
    __threadfence_block();
    const unsigned long long m = lane < 4 ? atomicExch(&mail[lane], kEmpty) : kEmpty;
    if (__any_sync(kFull, m != kEmpty)) {
      deliver(m != kEmpty ? 1u << lane : 0u, m);
      t0 = 0;
      continue;
    }
    if (__all_sync(kFull, over)) break;
    if ((it & 255u) == 255u) {
      int late = 0;
      if (lane == 0) {
        const long long now = now_ns();
        if (t0 == 0) t0 = now;
        late = now - t0 > limit;
        if (late) raise_status(p.ctl, kEtimeout, 8);
      }
      if (__shfl_sync(kFull, late, 0)) break;
    }
    __nanosleep(20);
  }
}

// AHEAD, HELP (2D): see above.
template <int D, bool AHEAD, bool HELP>
__global__ void __launch_bounds__(HELP ? 96 : 64, HELP ? kFrontCtasHelp : D == 3 ? kFrontCtas3 : AHEAD ? kFrontCtas2 : kFrontCtasMany2)
    front_kernel(SolveParams p) {
  constexpr int kAhead = 16;           // rounds a tile waits for its first front
  constexpr int TX = D == 3 ? 4 : 8, TY = TX, TZ = D == 3 ? 4 : 1, HZ = D == 3 ? 1 : 0;
  constexpr int SX = TX + 2, SY = TY + 2, SZ = TZ + 2 * HZ, NS = SX * SY * SZ;
  constexpr int F = 64 / TX, H = 2 * D * F, HW = H / 32, HT = (H + 63) / 64;   // cells per face, halo cells, words, per thread
  constexpr int kStride[3] = {1, SX, SX * SY};
  constexpr int kTile[3] = {TX, TY, TZ};
  struct Round {
    unsigned long long fmin[2];
    unsigned chg[2], hw[3], face[2];
  };
  __shared__ unsigned long long t_mem[NS];
  __shared__ Round flags[2];
  __shared__ unsigned long long sh_tile;
  __shared__ unsigned sh_lo, sh_slot;
  __shared__ int sh_faces;
  __shared__ unsigned long long mail[4];       // HELP: bucket time of a face to activate, kEmpty: none
  __shared__ volatile int sh_fin;              // HELP: the rounds are over
  volatile unsigned long long *const t = t_mem;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float inv_delta = static_cast<float>(p.ctl->inv_delta);
  long long idle_since = 0;
  auto pos_of = [](int x, int y, int z) { return ((z + HZ) * SY + y + 1) * SX + x + 1; };

  // this thread's cell and halo cells: the same in every tile
  const int cc[3] = {tid % TX, (tid / TX) % TY, tid / (TX * TY)};
  const int ps = pos_of(cc[0], cc[1], cc[2]);
  unsigned long long nb = 0ull;                         // in-tile neighbours
  unsigned hm[HW];                                      // halo neighbours
  unsigned edge = 0u;                                   // faces the cell lies on
#pragma unroll
  for (int c = 0; c < HW; ++c) hm[c] = 0u;
#pragma unroll
  for (int j = 0; j < 2 * D; ++j) {
    const int ax = j >> 1, d = ax == 0 ? 1 : ax == 1 ? TX : TX * TY;
    if (cc[ax] != ((j & 1) ? kTile[ax] - 1 : 0)) {
      nb |= 1ull << ((j & 1) ? tid + d : tid - d);
    } else {
      const int m = ax == 0 ? cc[1] + TY * cc[2] : ax == 1 ? cc[0] + TX * cc[2] : cc[0] + TX * cc[1];
      edge |= 1u << j;
      hm[j * F / 32] |= 1u << ((j * F + m) % 32);
    }
  }
  int hc[HT][3], hps[HT];
#pragma unroll
  for (int c = 0; c < HT; ++c) {
    const int i = c * 64 + tid, j = i / F, m = i % F, ax = j >> 1, e = (j & 1) ? kTile[ax < 3 ? ax : 0] : -1;
    hc[c][0] = ax == 0 ? e : m % TX;
    hc[c][1] = ax == 0 ? m % TY : ax == 1 ? e : m / TX;
    hc[c][2] = ax == 2 ? e : D == 3 ? m / TX : 0;
    hps[c] = i < H ? pos_of(hc[c][0], hc[c][1], hc[c][2]) : 0;
  }

  auto sync_rounds = [] {                      // the warps that hold cells
    if (HELP) asm volatile("bar.sync 1, 64;" ::: "memory");
    else __syncthreads();
  };
  if (HELP && tid < 4) mail[tid] = kEmpty;
  if (HELP && tid == 0) sh_fin = 0;
#pragma unroll 1
  for (;;) {
    if (warp == (HELP ? 2 : 0)) {
      unsigned slot = 0, lo = 0;
      unsigned long long tile = kEmpty;
      int faces = 0;
#pragma unroll 1
      for (;;) {
        const unsigned long long e = pop_entry(p, idle_since, slot, lo);
        if (e == kEmpty) break;
        const unsigned long long tl = e & 0xffffffffull;
        int f = -1;
        if (lane == 0) f = try_claim(p, tl, static_cast<unsigned>(e >> 32));
        f = __shfl_sync(kFull, f, 0);
        if (f >= 0) { tile = tl; faces = f; break; }
        if (lane == 0) {
          atomicAdd(&p.ctl->run[slot * kCounterPad], 0xffffffffu);
          atomicAdd(&p.ctl->work, -1);
        }
      }
      idle_since = 0;
      if (lane == 0) {
        fence_ar();    // the claim is ordered before the tile's loads
        sh_tile = tile;
        sh_lo = lo;
        sh_slot = slot;
        sh_faces = faces;
      }
    }
    __syncthreads();
    if (sh_tile == kEmpty) break;
    const long long tile = static_cast<long long>(sh_tile);
    const unsigned lo = sh_lo;
    const int faces = sh_faces;
    const Prob &P = p.probs[find_prob_ro(p, static_cast<unsigned>(tile))];
    const int64_t nx = ldg_i64(&P.nx), ny = ldg_i64(&P.ny), nz = ldg_i64(&P.nz);
    const unsigned ntx = static_cast<unsigned>(ldg_i64(&P.ntx)), nty = static_cast<unsigned>(ldg_i64(&P.nty)),
                   ntz = static_cast<unsigned>(ldg_i64(&P.ntz));
    const double *const C0 = reinterpret_cast<const double *>(ldg_i64(&P.c));
    unsigned tcx, tcy, tcz;
    {   // fewer than 2^32 tiles: 32-bit divisions
      const unsigned lt = static_cast<unsigned>(tile - ldg_i64(&P.tile_base));
      const unsigned rest = lt / ntx;
      tcx = lt - rest * ntx;
      tcz = rest / nty;
      tcy = rest - tcz * nty;
    }
    const int64_t x0 = static_cast<int64_t>(tcx) * TX, y0 = static_cast<int64_t>(tcy) * TY,
                  z0 = static_cast<int64_t>(tcz) * TZ;
    const int64_t sy = nx, sz = nx * ny, first = z0 * sz + y0 * sy + x0;
    unsigned long long *const T0 = reinterpret_cast<unsigned long long *>(ldg_i64(&P.t)) + first;
    // the faces across which there is a tile, and those of them this cell lies on
    const unsigned open_all = ((tcx > 0 ? 1u : 0u) | (tcx + 1 < ntx ? 2u : 0u) | (tcy > 0 ? 4u : 0u) |
                                  (tcy + 1 < nty ? 8u : 0u) | (tcz > 0 ? 16u : 0u) | (tcz + 1 < ntz ? 32u : 0u));
    const unsigned open = edge & ((tcx > 0 ? 1u : 0u) | (tcx + 1 < ntx ? 2u : 0u) | (tcy > 0 ? 4u : 0u) |
                                  (tcy + 1 < nty ? 8u : 0u) | (tcz > 0 ? 16u : 0u) | (tcz + 1 < ntz ? 32u : 0u));
    auto activate_faces = [&](unsigned set, unsigned long long min) {
      if ((set >> lane) & 1u) {
        fence_ar();
        const int64_t step = (lane >> 1) == 0 ? 1 : (lane >> 1) == 1 ? ntx : static_cast<int64_t>(ntx) * nty;
        activate(p, static_cast<unsigned long long>(tile + ((lane & 1) ? step : -step)), 1u << (lane ^ 1),
                 bucket_of_time(min, inv_delta), lo);
      }
      __syncwarp();
    };
    // done, unless the tile was re-activated meanwhile (one thread)
    auto finish = [&] { sh_faces = end_visit(p, static_cast<unsigned long long>(tile)); };
    if (HELP && warp == 2) {
#pragma unroll 1
      for (;;) {
        serve_mail(mail, &sh_fin, p, activate_faces);
        __syncwarp();
        if (lane == 0) {
          finish();
          sh_fin = 0;
        }
        __syncthreads();
        if (!sh_faces) break;
      }
      __syncthreads();
      continue;
    }
    const bool in = cc[0] < nx - x0 && cc[1] < ny - y0 && cc[2] < nz - z0;
    const int64_t off = cc[2] * sz + cc[1] * sy + cc[0];
    unsigned long long *const at = T0 + off;
    const unsigned long long c = in ? static_cast<unsigned long long>(ldg_i64(C0 + first + off)) : 0ull;
    {
      const unsigned long long v = in ? ld_rlx(at) : kInfBits;
      t[ps] = v;
      const unsigned b = __ballot_sync(kFull, v < kInfBits);
      if (lane == 0) flags[0].chg[warp] = b;
    }
    const bool fixed = !in || (p.tile_src[tile] != 0 && is_source(P, first + off));
    const unsigned long long *hat[HT];
    Round *fl = &flags[0];
#pragma unroll
    for (int h = 0; h < HT; ++h) {
      if (h * 64 + warp * 32 >= H) { hat[h] = nullptr; continue; }
      const int64_t x = x0 + hc[h][0], y = y0 + hc[h][1], z = z0 + hc[h][2];
      const bool hin = x >= 0 && x < nx && y >= 0 && y < ny && z >= 0 && z < nz;
      hat[h] = hin ? T0 + hc[h][2] * sz + hc[h][1] * sy + hc[h][0] : nullptr;
      const unsigned long long v = hin ? ld_rlx(hat[h]) : kInfBits;
      t[hps[h]] = v;
      const unsigned b = __ballot_sync(kFull, v < kInfBits);
      if (lane == 0) fl->hw[h * 2 + warp] = b;
    }
    sync_rounds();
    ig::Scaled<D> scaled;
    bool pend = (faces & (1 << kFaceFull)) != 0;
#pragma unroll
    for (int w = 0; w < HW; ++w) pend = pend || (hm[w] & fl->hw[w]) != 0u;
    pend = pend && !fixed;
    bool fresh = AHEAD && !(fl->chg[0] | fl->chg[1]);   // no front has reached the tile
    unsigned fin[HW];                                   // halo cells that have a value
#pragma unroll
    for (int w = 0; w < HW; ++w) fin[w] = fl->hw[w];
    int quiet = 0;
    unsigned notified = 0u, later = 0u;
    unsigned long long later_min = kInfBits;
    auto notify = [&](unsigned set, unsigned long long min) {    // warp 0
      if constexpr (HELP) {
        if ((set >> lane) & 1u) {
          __threadfence_block();
          atomicExch(&mail[lane & 3], min);
        }
        __syncwarp();
      } else {
        activate_faces(set, min);
      }
    };
    // the first front reaches the tile: the tiles that it has not reached either start
    // now, and look for it while it crosses this one
    auto wake = [&]() {
      unsigned set = 0u;
#pragma unroll
      for (int j = 0; j < 2 * D; ++j)
        if (!((fin[j * F / 32] >> (j * F % 32)) & ((1u << F) - 1u))) set |= 1u << j;
      set &= open_all;
      if (set && warp == 0) {
        unsigned long long m = kInfBits;      // the smallest halo value
#pragma unroll
        for (int w = 0; w < HW; ++w) {
          const int i = w * 32 + lane, j = i / F, n = i % F, ax = j >> 1, e = (j & 1) ? TX : -1;
          m = umin64(m, t[pos_of(ax == 0 ? e : n % TX, ax == 0 ? n % TY : ax == 1 ? e : n / TX,
                                 ax == 2 ? e : D == 3 ? n / TX : 0)]);
        }
        notify(set, warp_min64(m));
      }
      notified |= set;
    };
    if (fresh) {
      unsigned a = 0u;
#pragma unroll
      for (int w = 0; w < HW; ++w) a |= fin[w];
      if (a) { wake(); fresh = false; }
    }
#pragma unroll 1
    for (unsigned round = 0;; ++round) {
      if (round >= kMaxRounds) {
        if (tid == 0) raise_status(p.ctl, kEtimeout, 7);
        if (!HELP) break;
      }
      unsigned long long hv[HT];
#pragma unroll
      for (int h = 0; h < HT; ++h) hv[h] = hat[h] ? ld_rlx(hat[h]) : kInfBits;
      unsigned low = 0u;
      unsigned long long nv = kInfBits;
      bool did = false;
      if (__any_sync(kFull, pend)) {
        unsigned long long a[D], side[2 * D];
        const unsigned long long own = t[ps];
#pragma unroll
        for (int ax = 0; ax < D; ++ax) {
          side[2 * ax] = t[ps - kStride[ax]];
          side[2 * ax + 1] = t[ps + kStride[ax]];
          a[ax] = umin64(side[2 * ax], side[2 * ax + 1]);
        }
        if (pend) did = hw::relax<D>(own, a, c, nv, nullptr, scaled);
        __syncwarp();
        if (did) {
          t[ps] = nv;
          st_rlx(at, nv);
        }
#pragma unroll
        for (int j = 0; j < 2 * D; ++j) low |= (nv < side[j] ? 1u : 0u) << j;
        low = did ? low & open : 0u;
      }
      fl = &flags[(round & 1u) ^ 1u];
      {
        const unsigned b = __ballot_sync(kFull, did), f = __reduce_or_sync(kFull, low);
        if (lane == 0) { fl->chg[warp] = b; fl->face[warp] = f; }
        if (f) {
          const unsigned long long m = warp_min64(low ? nv : kInfBits);
          if (lane == 0) fl->fmin[warp] = m;
        }
      }
#pragma unroll
      for (int h = 0; h < HT; ++h) {
        if (h * 64 + warp * 32 >= H) continue;
        const bool fell = hv[h] < t[hps[h]];
        if (fell) t[hps[h]] = hv[h];
        const unsigned b = __ballot_sync(kFull, fell);
        if (lane == 0) fl->hw[h * 2 + warp] = b;
      }
      sync_rounds();
      const unsigned long long chg = (static_cast<unsigned long long>(fl->chg[1]) << 32) | fl->chg[0];
      unsigned any = fl->chg[0] | fl->chg[1];
      pend = (nb & chg) != 0ull;
#pragma unroll
      for (int w = 0; w < HW; ++w) {
        any |= fl->hw[w];
        pend = pend || (hm[w] & fl->hw[w]) != 0u;
      }
      pend = pend && !fixed;
      const unsigned f0 = fl->face[0], f1 = fl->face[1], bits = f0 | f1;
      if (bits) {
        const unsigned long long m = umin64(f0 ? fl->fmin[0] : kInfBits, f1 ? fl->fmin[1] : kInfBits);
        const unsigned now = bits & ~notified;
        if (bits & notified) later_min = umin64(later_min, m);
        later |= bits & notified;
        if (now && warp == 0) notify(now, m);
        notified |= now;
      }
      if (fresh) {
        unsigned a = 0u;
#pragma unroll
        for (int w = 0; w < HW; ++w) a |= (fin[w] |= fl->hw[w]);
        if (a) { wake(); fresh = false; }
      }
      if (any && (!HELP || round < kMaxRounds)) { quiet = 0; continue; }
      if (fresh && ++quiet <= kAhead) continue;
      if (warp == 0) {
        if (later) notify(later, later_min);
        if (HELP) {
          __threadfence_block();
          if (lane == 0) sh_fin = 1;
        } else if (lane == 0) {
          finish();
        }
      }
      later = 0u;
      later_min = kInfBits;
      __syncthreads();
      if (!sh_faces) break;
    }
    if (tid == 0) {
      atomicAdd(&p.ctl->run[sh_slot * kCounterPad], 0xffffffffu);
      atomicAdd(&p.ctl->work, -1);
    }
    __syncthreads();
  }
}

}  // namespace

cudaError_t launch_front(const SolveParams &p, int grid, cudaStream_t stream) {
  note_launches(1);
  if (p.ndim == 3) front_kernel<3, false, false><<<grid, 64, 0, stream>>>(p);
  else if (p.ahead == 2) front_kernel<2, true, true><<<grid, 96, 0, stream>>>(p);
  else if (p.ahead) front_kernel<2, true, false><<<grid, 64, 0, stream>>>(p);
  else front_kernel<2, false, false><<<grid, 64, 0, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace eik
