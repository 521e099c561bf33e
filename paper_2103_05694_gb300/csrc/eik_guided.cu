// Guided tile kernel: lean solves with automatic options of 3D batches large
// enough to fill the device with ordered work (the others: eik_front.cu).
//
// The asynchronous tile schedule of eik_solver.cu (same buckets, claims and
// activations) with another way to relax a claimed tile.  That kernel finds
// the order of a tile's cells by exact arithmetic: every round of provisional
// d-bar values costs two block barriers and a dependent chain, and a cell is
// evaluated 6 (3D batch) to 33 times (2D section).  Here one warp owns a tile
// and a visit has two parts:
//
//  1. Order.  The tile's values and halo become float offsets g from their
//     minimum, and the first-order update is relaxed in FP32 until nothing falls
//     by more than a thousandth of a cell's r (a row of 32 cells takes about 80
//     warp instructions).
//  2. Exact.  Each cell that may change is evaluated by d-bar once, after its
//     neighbours in the tile with smaller g.  The order is kept as bit sets over
//     the tile (one 32-bit word per lane): a cell is ready when none of the
//     neighbours it waits for is left in the set of cells to do, a handful of
//     shifts and masks per round for the whole tile, and the ready cells are
//     packed onto the lanes.
//  Then every cell is checked against the neighbours it did not wait for: one
//  that fell below it since makes it be evaluated again, until there are none.
//
// g only orders the evaluations.  When the visit ends, no neighbour has fallen
// below a cell since the cell's last evaluation, so the fixed point and its
// bits are those of any schedule (Theorem 1), whatever the floats say.  Nothing
// is deferred inside a visit: the look-ahead window only limits which tiles are
// taken.
//
// What bounds it: instructions (88-problem 3D batch: issue 52 % at 4.75 warps per
// scheduler, the instruction cache close to its request rate, so loops are rolled
// and the scheduler's functions are not inlined: 218 -> 75 ms for the 128-source
// batch).  Evaluations per cell: 2.5 against 6.1 in the kernel of eik_solver.cu.
// Measured against that kernel with the same d-bar: 88-problem batch 115.7 -> 57.4
// ms.  Tiles: 8x8x4 70 ms, 8x4x4 88 ms, 4x4x4 113 ms (an earlier state).
// Tried and dropped: a visit limit inside the tile (narrow windows leave partial
// tiles: batch 75 -> 139 ms at a quarter of the bucket width); waiting while a
// neighbour tile is being visited (visits halve, the wait costs more); skipping
// cells no neighbour has fallen below (batch 71.7 -> 74.1 ms); more warps per SM
// with fewer registers (69.0 -> 73.5 ms at 23).
#include <cstdint>
#include <cuda_runtime.h>

#include "eik_exact.cuh"
#include "eik_internal.h"
#define EIK_SCHED_FN __device__ __noinline__   // one copy each: the kernel is bound by instruction fetch
#include "eik_sched.cuh"

namespace eik {
namespace {

constexpr float kSettled = 1e-3f;   // falls below this many r stop the FP32 relaxation

// (v - base) times 2^-se as a float for bit patterns v >= base >= 0, without the
// FP64 pipe: the significands' integer difference where v lies within 8
// binades of base, else the difference of the floats.
__device__ __forceinline__ float offset_f(unsigned long long v, unsigned long long base, int se) {
  constexpr unsigned long long kFrac = (1ull << 52) - 1, kHid = 1ull << 52;
  const int eb = static_cast<int>(base >> 52), d = static_cast<int>(v >> 52) - eb;
  if (eb == 0 || d > 8) return to_f_scaled(v, se) - (v < kInfBits ? to_f_scaled(base, se) : 0.0f);
  const unsigned long long x = (((v & kFrac) | kHid) << d) - ((base & kFrac) | kHid);
  const float f = fmaf(__uint2float_rn(static_cast<unsigned>(x >> 32)), 4294967296.0f,
                       __uint2float_rn(static_cast<unsigned>(x)));
  const int e = eb - 1075 - se;                   // unit 2^(eb - 1075)
  const int e1 = e < -126 ? -126 : e > 126 ? 126 : e, e2 = e - e1 < -126 ? -126 : e - e1;
  return f * __int_as_float((127 + e1) << 23) * __int_as_float((127 + (e2 > 0 ? 126 : e2)) << 23);
}

// First-order update in FP32 from the axis minima (offsets; +inf allowed), r = h / v.
__device__ __forceinline__ float root_f(const float (&a)[3], float r) {
  float lo = fminf(a[0], a[1]), hi = fmaxf(a[0], a[1]);
  const float top = fmaxf(hi, a[2]), m = fminf(hi, a[2]);
  hi = fmaxf(lo, m);
  lo = fminf(lo, m);
  float u = r;
  const float b1 = hi - lo;               // NaN when both are +inf: one-sided
  if (b1 < r) {
    const float rr = r * r;
    u = 0.5f * (b1 + ffa::sqrt_est(fmaf(-b1, b1, 2.0f * rr)));
    const float b2 = top - lo;
    if (b2 < u) {
      const float s = b1 + b2, q = fmaf(b1, b1, b2 * b2);
      const float disc = fmaxf(fmaf(s, s, -3.0f * (q - rr)), 1e-30f);
      u = (s + ffa::sqrt_est(disc)) * (1.0f / 3.0f);
    }
  }
  return lo + u;
}

template <int TX, int TY, int TZ>
struct GTile {
  static constexpr int NT = TX * TY * TZ, NC = NT / 32;
  static constexpr int SX = TX + 2, SY = TY + 2, SZ = TZ + 2, NS = SX * SY * SZ;
  double t[NS];                    // exact values with halo
  unsigned long long c[NT];
  float g[NS];                     // predicted offsets with halo
  float r[NT];                     // h / v
  unsigned char list[NT];
  unsigned char fell[NT];          // 1: fell since the last look
};

template <int TX, int TY, int TZ>
__global__ void __launch_bounds__(32, kGuidedCtas) guided_kernel(SolveParams p) {
  using S = GTile<TX, TY, TZ>;
  constexpr int D = 3, NT = S::NT, NC = S::NC, SX = S::SX, SY = S::SY;
  static_assert(NT % 32 == 0 && NT <= 256, "whole warps, 8-bit list entries");
  constexpr int kStride[3] = {1, SX, SX * SY};
  constexpr int kTile[3] = {TX, TY, TZ};
  __shared__ S s;
  const int lane = threadIdx.x;
  const float inv_delta = static_cast<float>(p.ctl->inv_delta);
  const int se = p.ctl->scale_exp;
  long long idle_since = 0;
  auto pos_of = [](int q) { return ((q / (TX * TY) + 1) * SY + (q / TX) % TY + 1) * SX + q % TX + 1; };
  auto nbrs = [](unsigned w, int j) { return face_bits<TX, TY, TZ>(w, j); };

#pragma unroll 1
  for (;;) {
    long long tile = -1;
    int faces = 0;
    unsigned slot = 0, lo = 0;
#pragma unroll 1
    for (;;) {
      const unsigned long long e = pop_entry(p, idle_since, slot, lo);
      if (e == kEmpty) break;
      const unsigned long long tl = e & 0xffffffffull;
      int f = -1;
      if (lane == 0) f = try_claim(p, tl, static_cast<unsigned>(e >> 32));
      f = __shfl_sync(kFull, f, 0);
      if (f >= 0) { tile = static_cast<long long>(tl); faces = f; break; }
      if (lane == 0) {
        atomicAdd(&p.ctl->run[slot * kCounterPad], 0xffffffffu);
        atomicAdd(&p.ctl->work, -1);
      }
    }
    if (tile < 0) break;
    idle_since = 0;
    // the problem's record through the read-only path: the fence below would
    // send each of these dependent reads to L2
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
    double *const T0 = reinterpret_cast<double *>(ldg_i64(&P.t)) + first;   // the tile's first cell
    fence_ar();      // the claim is ordered before the tile's loads
    // the grid in tile coordinates, as far as the tile and its halo reach
    const int xlo = x0 > 0 ? -1 : 0, ylo = y0 > 0 ? -1 : 0, zlo = z0 > 0 ? -1 : 0;
    const int xhi = nx - x0 > TX ? TX + 1 : static_cast<int>(nx - x0);
    const int yhi = ny - y0 > TY ? TY + 1 : static_cast<int>(ny - y0);
    const int zhi = nz - z0 > TZ ? TZ + 1 : static_cast<int>(nz - z0);
    unsigned fixed_w = 0u;               // sources and cells off the grid: word k in lane k
    const bool has_src = p.tile_src[tile] != 0;
#pragma unroll 4
    for (int k = 0; k < NC; ++k) {
      const int q = k * 32 + lane;
      const int ix = q % TX, iy = (q / TX) % TY, iz = q / (TX * TY);
      const bool in = ix < xhi && iy < yhi && iz < zhi;
      const int64_t off = iz * sz + iy * sy + ix;
      const double tv = in ? ld_time(T0 + off) : from_bits(kInfBits);
      const unsigned long long cv =
          in ? static_cast<unsigned long long>(__ldg(reinterpret_cast<const long long *>(C0) + first + off)) : 0ull;
      s.t[pos_of(q)] = tv;
      s.c[q] = cv;
      s.fell[q] = 0;
      const float cf = to_f_scaled(cv, 2 * se);
      s.r[q] = cf > 0.0f ? ffa::sqrt_est(cf) : 0.0f;
      const unsigned b = __ballot_sync(kFull, !in);
      if (lane == k) fixed_w = b;
    }
    if (has_src) {
#pragma unroll 1
      for (int k = 0; k < NC; ++k) {
        const int q = k * 32 + lane;
        const unsigned b = __ballot_sync(kFull, is_source(P, first + (q / (TX * TY)) * sz + ((q / TX) % TY) * sy + q % TX));
        if (lane == k) fixed_w |= b;
      }
    }

    // A claimed tile is worked on until no neighbour has re-activated it meanwhile.
#pragma unroll 1
    for (;;) {
      {  // halo faces: y (x fastest: coalesced), z, x
        constexpr int FX = TY * TZ, FY = TX * TZ, FZ = TX * TY;
        constexpr int H = 2 * FX + 2 * FY + 2 * FZ;
#pragma unroll 4
        for (int i = lane; i < H; i += 32) {
          int ix, iy, iz;                // tile coordinates, -1 .. extent
          if (i < 2 * FY) {
            const int j = i % FY;
            ix = j % TX; iz = j / TX; iy = i < FY ? -1 : TY;
          } else if (i < 2 * FY + 2 * FZ) {
            const int k = i - 2 * FY, j = k % FZ;
            ix = j % TX; iy = j / TX; iz = k < FZ ? -1 : TZ;
          } else {
            const int k = i - 2 * FY - 2 * FZ, j = k % FX;
            iy = j % TY; iz = j / TY; ix = k < FX ? -1 : TX;
          }
          const bool in = ix >= xlo && ix < xhi && iy >= ylo && iy < yhi && iz >= zlo && iz < zhi;
          s.t[((iz + 1) * SY + iy + 1) * SX + ix + 1] =
              in ? ld_time(T0 + iz * sz + iy * sy + ix) : from_bits(kInfBits);
        }
      }
      __syncwarp();

      // cells to evaluate: every cell (a seeded tile), or those next to a changed
      // halo value that is below theirs
      unsigned need_w = (faces & (1 << kFaceFull)) ? kFull : 0u;
      unsigned long long base = kInfBits;
#pragma unroll 1
      for (int k = 0; k < NC; ++k) {
        const int q = k * 32 + lane, ps = pos_of(q);
        const int cc[3] = {q % TX, (q / TX) % TY, q / (TX * TY)};
        const unsigned long long tb = bits_of(s.t[ps]);
        bool want = false;
        base = umin64(base, tb);
#pragma unroll
        for (int j = 0; j < 2 * D; ++j) {
          const int ax = j >> 1;
          if (cc[ax] != ((j & 1) ? kTile[ax] - 1 : 0)) continue;
          const unsigned long long hv = bits_of(s.t[ps + ((j & 1) ? kStride[ax] : -kStride[ax])]);
          base = umin64(base, hv);
          want = want || (((faces >> j) & 1) && hv < tb);
        }
        const unsigned b = __ballot_sync(kFull, want);
        if (lane == k) need_w |= b;
      }
      need_w = lane < NC ? need_w & ~fixed_w : 0u;
      unsigned changed_w = 0u;
      if (__any_sync(kFull, need_w != 0u)) {
        base = warp_min64(base);
        // offsets from the smallest value, in units of 2^se
#pragma unroll 1
        for (int i = lane; i < S::NS; i += 32) s.g[i] = offset_f(bits_of(s.t[i]), base, se);
        unsigned fixed = 0u;                    // bit k: this lane's cell k
#pragma unroll
        for (int k = 0; k < NC; ++k) fixed |= ((__shfl_sync(kFull, fixed_w, k) >> lane) & 1u) << k;
        __syncwarp();
        // 1. order: relax in FP32 by rows of 32 cells, up and down by turns, each row
        // while one of its neighbour rows (or itself) has fallen since its last turn
        unsigned stale = (1u << NC) - 1u;
        static_assert(TX * TY == 64, "a slice is two rows");
#pragma unroll 1
        for (int it = 0; stale && it < 4 * NT; ++it) {
#pragma unroll 1
          for (int kk = 0; kk < NC; ++kk) {
            const int k = (it & 1) ? NC - 1 - kk : kk;
            if (!((stale >> k) & 1u)) continue;
            const int q = k * 32 + lane, ps = pos_of(q);
            float a[D];
#pragma unroll
            for (int ax = 0; ax < D; ++ax) a[ax] = fminf(s.g[ps - kStride[ax]], s.g[ps + kStride[ax]]);
            const float r = s.r[q];
            const float nv = root_f(a, r);
            const bool fell = !((fixed >> k) & 1u) && nv < s.g[ps] - kSettled * r;
            if (fell) s.g[ps] = nv;
            stale &= ~(1u << k);
            if (__any_sync(kFull, fell)) {
              // rows k, k +- 1 and, in the next slices, k +- 2
              stale |= (((7u << k) >> 1) | ((17u << k) >> 2)) & ((1u << NC) - 1u);
            }
            __syncwarp();
          }
        }
        // a cell that will be evaluated can change only cells of larger g
        float g_need = kInfF;
#pragma unroll 1
        for (int k = 0; k < NC; ++k)
          if ((__shfl_sync(kFull, need_w, k) >> lane) & 1u) g_need = fminf(g_need, s.g[pos_of(k * 32 + lane)]);
        g_need = __uint_as_float(__reduce_min_sync(kFull, __float_as_uint(g_need)));
        unsigned todo_w = 0u;                   // cells to evaluate
        unsigned up_w[2 * D];                   // cells that wait for their neighbour across face j
#pragma unroll
        for (int j = 0; j < 2 * D; ++j) up_w[j] = 0u;
#pragma unroll 1
        for (int k = 0; k < NC; ++k) {
          const int q = k * 32 + lane, ps = pos_of(q);
          const int cc[3] = {q % TX, (q / TX) % TY, q / (TX * TY)};
          const float gq = s.g[ps];
          const unsigned be = __ballot_sync(kFull, gq >= g_need && gq < kInfF);
          if (lane == k) todo_w = be;
#pragma unroll
          for (int j = 0; j < 2 * D; ++j) {
            const int ax = j >> 1;
            const unsigned b = __ballot_sync(kFull, cc[ax] != ((j & 1) ? kTile[ax] - 1 : 0) &&
                                                        s.g[ps + ((j & 1) ? kStride[ax] : -kStride[ax])] < gq);
            if (lane == k) up_w[j] = b;
          }
        }
        todo_w = (todo_w | need_w) & ~fixed_w;
#pragma unroll
        for (int j = 0; j < 2 * D; ++j) up_w[j] &= nbrs(todo_w, j) & todo_w;
        // 2. exact evaluations in that order
        bool ordered = true;
#pragma unroll 1
        for (unsigned round = 0;; ++round) {
          if (round >= kMaxRounds) {
            if (lane == 0) raise_status(p.ctl, kEtimeout, 7);
            break;
          }
          unsigned ready_w = todo_w;
          if (ordered) {
#pragma unroll
            for (int j = 0; j < 2 * D; ++j) ready_w &= ~(up_w[j] & nbrs(todo_w, j));
          }
          const int n = list_of_set<NC>(ready_w, s.list);
          __syncwarp();
          if (n > 0) {
            todo_w &= ~ready_w;
#pragma unroll 1
            for (int b = lane; b < ((n + 31) & ~31); b += 32) {
              if (b < n) {
                const int q = s.list[b], ps = pos_of(q);
                unsigned long long a[D];
                const unsigned long long best = bits_of(s.t[ps]);
#pragma unroll
                for (int ax = 0; ax < D; ++ax)
                  a[ax] = umin64(bits_of(s.t[ps - kStride[ax]]), bits_of(s.t[ps + kStride[ax]]));
                unsigned long long nv;
                if (hw::relax<D>(best, a, s.c[q], nv)) {
                  s.t[ps] = from_bits(nv);
                  s.fell[q] = 1;
                }
              }
            }
            __syncwarp();
            if (ordered) continue;
          }
          // All listed cells are evaluated.  A cell is right unless a neighbour it
          // did not wait for has fallen below it since: list those, in any order.
          unsigned now_w = 0u, redo_w = 0u, below_w[2 * D];
#pragma unroll
          for (int j = 0; j < 2 * D; ++j) below_w[j] = 0u;
#pragma unroll 1
          for (int k = 0; k < NC; ++k) {
            const int q = k * 32 + lane, ps = pos_of(q);
            const int cc[3] = {q % TX, (q / TX) % TY, q / (TX * TY)};
            const unsigned b = __ballot_sync(kFull, s.fell[q] != 0);
            s.fell[q] = 0;
            if (lane == k) now_w = b;
            const unsigned long long tb = bits_of(s.t[ps]);
#pragma unroll
            for (int j = 0; j < 2 * D; ++j) {
              const int ax = j >> 1;
              const unsigned bj = __ballot_sync(
                  kFull, cc[ax] != ((j & 1) ? kTile[ax] - 1 : 0) &&
                             bits_of(s.t[ps + ((j & 1) ? kStride[ax] : -kStride[ax])]) < tb);
              if (lane == k) below_w[j] = bj;
            }
          }
          changed_w |= now_w;
          if (!__any_sync(kFull, now_w != 0u)) break;
#pragma unroll
          for (int j = 0; j < 2 * D; ++j)
            redo_w |= below_w[j] & nbrs(now_w, j) & ~(ordered ? up_w[j] : 0u);
          todo_w = redo_w & ~fixed_w;
          ordered = false;
          if (!__any_sync(kFull, todo_w != 0u)) break;
        }
      }

      // commit, and the smallest committed time per face that is below the
      // halo value across it (only such a value can change the cell there)
      if (__any_sync(kFull, changed_w != 0u)) {
        unsigned fm_any = 0u;
        unsigned long long fm[2 * D];
#pragma unroll
        for (int j = 0; j < 2 * D; ++j) fm[j] = kInfBits;
#pragma unroll 1
        for (int k = 0; k < NC; ++k) {
          if (!((__shfl_sync(kFull, changed_w, k) >> lane) & 1u)) continue;
          const int q = k * 32 + lane, ps = pos_of(q);
          const int cc[3] = {q % TX, (q / TX) % TY, q / (TX * TY)};
          const unsigned long long tb = bits_of(s.t[ps]);
          // only this tile's visit writes its cells: a plain store
          st_rlx(reinterpret_cast<unsigned long long *>(T0 + cc[2] * sz + cc[1] * sy + cc[0]), tb);
#pragma unroll
          for (int j = 0; j < 2 * D; ++j) {
            const int ax = j >> 1;
            if (cc[ax] != ((j & 1) ? kTile[ax] - 1 : 0)) continue;
            if (tb < bits_of(s.t[ps + ((j & 1) ? kStride[ax] : -kStride[ax])])) fm[j] = umin64(fm[j], tb);
          }
        }
        unsigned long long mine = kInfBits;
#pragma unroll
        for (int j = 0; j < 2 * D; ++j) {
          if (!__any_sync(kFull, fm[j] < kInfBits)) continue;
          const unsigned long long v = warp_min64(fm[j]);
          if (lane == j) mine = v;
          fm_any |= 1u << j;
        }
        __syncwarp();
        fence_ar();               // every lane's stores before the activations
        if ((fm_any >> lane) & 1u) {
          const int ax = lane >> 1, up = lane & 1;
          const unsigned at = ax == 0 ? tcx : ax == 1 ? tcy : tcz, ext = ax == 0 ? ntx : ax == 1 ? nty : ntz;
          if (up ? at + 1 < ext : at > 0) {
            const int64_t step = ax == 0 ? 1 : ax == 1 ? ntx : static_cast<int64_t>(ntx) * nty;
            activate(p, static_cast<unsigned long long>(tile + (up ? step : -step)), 1u << (lane ^ 1),
                     bucket_of_time(mine, inv_delta), lo);
          }
        }
        __syncwarp();
      }
      // done, unless the tile was re-activated meanwhile: then go on with its new
      // faces
      int cont = 0;
      if (lane == 0) cont = end_visit(p, static_cast<unsigned long long>(tile));
      cont = __shfl_sync(kFull, cont, 0);
      if (!cont) break;
      faces = cont & 0x7f;
    }

    if (lane == 0) {
      atomicAdd(&p.ctl->run[slot * kCounterPad], 0xffffffffu);
      atomicAdd(&p.ctl->work, -1);
    }
    __syncwarp();
  }
}

}  // namespace

cudaError_t launch_guided(const SolveParams &p, int grid, cudaStream_t stream) {
  note_launches(1);
  guided_kernel<8, 8, 4><<<grid, 32, 0, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace eik
