// Adjoint of the exact fixed point: d(loss)/d(slowness) for traveltime
// tomography (not in the paper; implicit differentiation of the
// real-arithmetic local equations at the computed field).
//
// For a reached non-source cell n with axis minima a_k and active axes
// A(n) = {k : a_k < t_n}, the local equation sum_{k in A} (t_n - a_k)^2 =
// h^2 s_n^2 (s = 1/v) gives dt_n = [sum_A (t_n - a_k) da_k + h^2 s_n ds_n] / S_n
// with S_n = sum_A (t_n - a_k).  For g = dL/dt:
//   lambda_n = g_n + sum_{downwind m, order x-, x+, y-, y+, z-, z+} lambda_m w(m, n),
//   w(m, n)  = (t_m - t_n) / S_m, halved when m's two neighbours on that axis tie,
//   dL/ds_n  = lambda_n (h^2 s_n) / S_n   (0 for sources and unreached cells).
// Every operation is an explicit round-to-nearest intrinsic and the sum order
// is fixed, so the result equals the CPU oracle's bit for bit.
//
// Set-up (fully parallel) evaluates everything that does not depend on lambda:
// per cell m the mask of its upwind sides, the weight of each active axis
// W_k(m) = fl(fl(t_m - a_k) / S_m) (halved on a tie) and the coefficient
// fl(fl(h^2 fl(1 / v)) / S).  The dependent part is then one multiply-add per
// downwind neighbour.
//
// Two schedules process the cells in dependency (Kahn) order with the same
// operations in the same order, so their results are identical:
//  * tiles (the default; see "Tile schedule" below): persistent warps take
//    tiles from the bucket scheduler and run the order inside a tile in shared
//    memory, handing cross-tile dependencies over through the cells' mask bytes;
//  * levels: the set-up also counts every cell's downwind users; cells with count 0 form the first frontier; one cooperative
//    persistent launch processes a frontier (each cell pulls lambda from its
//    downwind cells, writes lambda and dL/ds, decrements its upwind cells'
//    counts and appends those that reach zero to the next frontier), then its
//    blocks meet at a grid barrier bounded by %globaltimer.  (Letting a thread
//    follow the cells it releases does not pay on this graph: in 2D most cells
//    have two downwind users, so chains merge after about two steps while the
//    few long chains stretch every frontier.)
#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

#include "eik_exact.cuh"
#include "eik_grid.cuh"
#include "eik_internal.h"
#define EIK_SCHED_FN __device__ __noinline__
#define EIK_SCHED_PROGRESS 1
#include "eik_sched.cuh"

namespace eik {
namespace {

constexpr unsigned long long kInfB = 0x7ff0000000000000ull;
constexpr unsigned kFullMask = 0xffffffffu;
constexpr int kThreads = 1024;   // threads per block of the level kernel

__device__ __forceinline__ unsigned long long ubits(double x) {
  return static_cast<unsigned long long>(__double_as_longlong(x));
}
__device__ __forceinline__ double ld_rlx_d(const double *p) {
  double v;
  asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long ld_rlx_u64(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_rlx_d(double *p, double v) {
  asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}

__device__ __forceinline__ int find_adj_prob(const AdjProb *probs, int nprob, int64_t q) {
  int lo = 0, hi = nprob - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (probs[mid].base <= q) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ bool adj_is_source(const AdjProb &P, int64_t n) {
  int64_t lo = 0, hi = P.nsrc - 1;
  while (lo <= hi) {
    const int64_t mid = (lo + hi) >> 1;
    const int64_t v = P.src_idx[mid];
    if (v == n) return true;
    if (v < n) lo = mid + 1; else hi = mid - 1;
  }
  return false;
}

// A cell with its coordinates, so that neighbours need no division.
struct Cell {
  int64_t n;
  int64_t c[3];
};

__device__ __forceinline__ Cell cell_of(const AdjProb &P, int64_t n) {
  Cell e;
  e.n = n;
  if (P.nx * P.ny * P.nz < (int64_t(1) << 31)) {     // 32-bit division where it fits
    const unsigned un = static_cast<unsigned>(n), ux = static_cast<unsigned>(P.nx),
                   uy = static_cast<unsigned>(P.ny);
    const unsigned yz = un / ux;
    e.c[0] = static_cast<int64_t>(un - yz * ux);
    e.c[1] = static_cast<int64_t>(yz % uy);
    e.c[2] = static_cast<int64_t>(yz / uy);
    return e;
  }
  const int64_t yz = n / P.nx;
  e.c[0] = n - yz * P.nx;
  e.c[1] = yz % P.ny;
  e.c[2] = yz / P.ny;
  return e;
}

// A frontier entry: problem index above bit kEntryShift, cell index below.
constexpr int kEntryShift = 40;
__device__ __forceinline__ unsigned long long entry_of(int pi, int64_t n) {
  return (static_cast<unsigned long long>(pi) << kEntryShift) | static_cast<unsigned long long>(n);
}

// Neighbour of a cell on side j (0..5: x-, x+, y-, y+, z-, z+), -1 off the grid.
__device__ __forceinline__ int64_t nbr(const AdjProb &P, const Cell &e, int j) {
  const int k = j >> 1;
  if (k >= P.ndim) return -1;
  const int64_t ext = k == 0 ? P.nx : (k == 1 ? P.ny : P.nz);
  const int64_t st = k == 0 ? 1 : (k == 1 ? P.nx : P.nx * P.ny);
  if (j & 1) return e.c[k] + 1 < ext ? e.n + st : -1;
  return e.c[k] > 0 ? e.n - st : -1;
}

// Per cell: the upwind-side mask, per-axis weights, and the gradient coefficient
// (kept in grad until lambda is known).
constexpr unsigned kPending = 0x40u, kDone = 0x80u;   // tile schedule: in the mask byte

// fl(h^2 s) of a cell, s = fl(1/v); slowness input: v = fl(1/s_in) as the forward used.
__device__ __forceinline__ double h2s(double v, int v_is_slowness, double hh) {
  const double vn = v_is_slowness ? ig::quotient(1.0, v) : v;
  return __dmul_rn(hh, ig::quotient(1.0, vn));
}

// The same for a whole model that several problems share: the set-up is bound
// by its divisions, of which a slowness model needs two here, and per problem one
// per active axis and one for the coefficient.  32 problems of 1024^2 cells on one
// model: set-up and this kernel 2.70 -> 1.9 ms by sharing (and a grid row per
// problem in place of a search per cell), 1.02 ms with the divisions off the FP64
// pipe (ig::Divisor).
__global__ void adj_h2s_kernel(const double *__restrict__ v, int v_is_slowness, double hh, int64_t n,
                               double *__restrict__ hs) {
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    hs[i] = h2s(v[i], v_is_slowness, hh);
}

// Mask, weights and coefficient of cell n with time tn; returns the mask.
template <bool COUNT>
__device__ __forceinline__ unsigned setup_cell(const AdjProb &P, int64_t n, double tn) {
  double coef = 0.0;
  unsigned mask = 0u;
  if (ubits(tn) < kInfB && !(P.nsrc > 0 && adj_is_source(P, n))) {
    const Cell e = cell_of(P, n);
    unsigned long long lo[3], hi[3], ak[3];
    double d[3], S = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (k >= P.ndim) break;
      const int64_t a = nbr(P, e, 2 * k), b = nbr(P, e, 2 * k + 1);
      lo[k] = a >= 0 ? ubits(P.t[a]) : kInfB;
      hi[k] = b >= 0 ? ubits(P.t[b]) : kInfB;
      ak[k] = lo[k] < hi[k] ? lo[k] : hi[k];
      if (ak[k] < ubits(tn)) {
        d[k] = __dsub_rn(tn, __longlong_as_double(static_cast<long long>(ak[k])));
        S = __dadd_rn(S, d[k]);
      }
    }
    if (S > 0.0) {   // else unreachable for a reached non-source cell
      const ig::Divisor by_S(ubits(S));
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (k >= P.ndim) break;
        if (!(ak[k] < ubits(tn))) continue;               // axis not active
        double w = __longlong_as_double(static_cast<long long>(by_S.quotient(ubits(d[k]))));
        if (lo[k] == hi[k]) w = __dmul_rn(w, 0.5);        // tie: half to each side
        P.W[k][n] = w;
        if (lo[k] == ak[k]) mask |= 1u << (2 * k);
        if (hi[k] == ak[k]) mask |= 1u << (2 * k + 1);
        if (COUNT) {
          if (lo[k] == ak[k]) atomicAdd(P.cnt + nbr(P, e, 2 * k), 1);
          if (hi[k] == ak[k]) atomicAdd(P.cnt + nbr(P, e, 2 * k + 1), 1);
        }
      }
      coef = __longlong_as_double(static_cast<long long>(
          by_S.quotient(ubits(P.hs ? P.hs[n] : h2s(P.v[n], P.v_is_slowness, P.hh)))));
    }
  }
  P.grad[n] = coef;
  return mask;
}

// Level schedule: also zeroed lambda and the downwind-use counts of the upwind cells.
__global__ void adj_setup_kernel(const AdjProb *probs, int nprob, int64_t total, AdjCtl *ctl) {
  unsigned long long reached = 0;
  for (int64_t q = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; q < total;
       q += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const AdjProb &P = probs[find_adj_prob(probs, nprob, q)];
    const int64_t n = q - P.base;
    const double tn = P.t[n];
    reached += ubits(tn) < kInfB ? 1u : 0u;
    P.lam[n] = 0.0;
    P.mask[n] = static_cast<unsigned char>(setup_cell<true>(P, n, tn));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) reached += __shfl_xor_sync(kFullMask, reached, o);
  if ((threadIdx.x & 31) == 0 && reached) atomicAdd(&ctl->reached, reached);
}

// The cells of all problems, shared out for the set-up and the search for ready cells.
// rows: a grid row per problem (first + blockIdx.y), so that no cell searches for
// its problem.  Else one loop over all cells, which looks the problem up where it
// changes: a row per problem gives each as many blocks as the average one needs, so
// a batch whose largest problem is far above the average waits for that one (call
// without the host's part, rows and one loop: a 256^3 volume beside 100 grids of
// 20 x 21 x 22 27.9 and 8.8 ms, 3000^2 beside 200 of 40 x 50 26.1 and 9.5 to 11.2),
// while like problems gain by the rows (3000 of 30 x 30, the same cells in equal
// pieces of the loop: 0.53 and 0.57 ms, 2000 of 5 x 6 0.10 and 0.15).
// cell(P, n) for each cell, leave(P) after a thread's last cell of P (rows: all
// threads of a block together).
template <class Cells, class Leave>
__device__ __forceinline__ void for_cells(const AdjProb *probs, int nprob, int64_t total, int first, bool rows,
                                          Cells cell, Leave leave) {
  const int64_t at = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x,
                step = static_cast<int64_t>(gridDim.x) * blockDim.x;
  if (rows) {
    const AdjProb &P = probs[first + blockIdx.y];
    const int64_t cells = P.nx * P.ny * P.nz;
    for (int64_t n = at; n < cells; n += step) cell(P, n);
    leave(P);
    return;
  }
  for (int64_t q = at; q < total;) {
    const AdjProb &P = probs[find_adj_prob(probs, nprob, q)];
    const int64_t end = P.base + P.nx * P.ny * P.nz;
    for (; q < end; q += step) cell(P, q - P.base);
    leave(P);
  }
}

// Tile schedule: the mask byte carries kPending (reached), and the problem's
// largest time is collected (the tiles' order), with one atomic per warp where the
// warp is of one problem; else only by those above what is there.
template <bool ROWS>
__global__ void adj_setup_tiles_kernel(const AdjProb *probs, int nprob, int64_t total, int first, AdjCtl *ctl) {
  unsigned long long reached = 0;
  unsigned top = 0u;        // high word of the largest finite time
  for_cells(probs, nprob, total, first, ROWS, [&](const AdjProb &P, int64_t n) {
    const double tn = P.t[n];
    const bool is_reached = ubits(tn) < kInfB;
    if (is_reached) {
      ++reached;
      const unsigned hi = static_cast<unsigned>(ubits(tn) >> 32);
      top = top < hi ? hi : top;
    }
    P.mask[n] = static_cast<unsigned char>(setup_cell<false>(P, n, tn) | (is_reached ? kPending : 0u));
  }, [&](const AdjProb &P) {
    if (ROWS) {
      const unsigned m = __reduce_max_sync(kFullMask, top);
      top = (threadIdx.x & 31) == 0 ? m : 0u;
    }
    const unsigned long long v = static_cast<unsigned long long>(top) << 32;
    if (top && v > ld_rlx_u64(P.tmax)) atomicMax(P.tmax, v);
    top = 0u;
  });
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) reached += __shfl_xor_sync(kFullMask, reached, o);
  if ((threadIdx.x & 31) == 0 && reached) atomicAdd(&ctl->reached, reached);
}

// Warp-aggregated append of the lanes' ready entries to a frontier.  All 32
// lanes of the warp call it.
__device__ __forceinline__ void append_ready(unsigned long long *count, unsigned long long *front,
                                             bool ready, unsigned long long entry) {
  const unsigned bal = __ballot_sync(kFullMask, ready);
  if (!bal) return;
  const unsigned lane = threadIdx.x & 31u;
  const int leader = __ffs(bal) - 1;
  unsigned long long base = 0;
  if (lane == static_cast<unsigned>(leader))
    base = atomicAdd(count, static_cast<unsigned long long>(__popc(bal)));
  base = __shfl_sync(kFullMask, base, leader);
  if (ready) front[base + __popc(bal & ((1u << lane) - 1u))] = entry;
}

__global__ void adj_seed_kernel(const AdjProb *probs, int nprob, int64_t total, AdjCtl *ctl,
                                unsigned long long *front) {
  const int64_t span = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t base = blockIdx.x * static_cast<int64_t>(blockDim.x); base < total; base += span) {
    const int64_t q = base + threadIdx.x;
    bool ready = false;
    unsigned long long ent = 0;
    if (q < total) {
      const int pi = find_adj_prob(probs, nprob, q);
      const AdjProb &P = probs[pi];
      const int64_t n = q - P.base;
      ready = ubits(P.t[n]) < kInfB && P.cnt[n] == 0;
      ent = entry_of(pi, n);
    }
    append_ready(&ctl->nfront[0], front, ready, ent);
  }
}

// lambda and dL/ds of one ready cell, then release its upwind cells; the ones
// that become ready are appended to the next frontier.  All 32 lanes call it.
__device__ void adj_process(const AdjProb *probs, unsigned long long entry, bool live,
                            unsigned long long *count, unsigned long long *front) {
  unsigned long long ready_entry[6];
  bool ready[6] = {false, false, false, false, false, false};
  if (live) {
    const int pi = static_cast<int>(entry >> kEntryShift);
    const AdjProb &P = probs[pi];
    const Cell e = cell_of(P, static_cast<int64_t>(entry & ((1ull << kEntryShift) - 1ull)));
    const int64_t n = e.n;
    int64_t m[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) m[j] = nbr(P, e, j);
    unsigned mm[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) mm[j] = m[j] >= 0 ? P.mask[m[j]] : 0u;
    double lam = P.g ? P.g[n] : 0.0;
    // pull from the downwind neighbours m for which n is an upwind side
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      if (!((mm[j] >> (j ^ 1)) & 1u)) continue;          // n is m's side j^1
      const double lm = ld_rlx_d(P.lam + m[j]);           // written by another thread
      lam = __dadd_rn(lam, __dmul_rn(lm, P.W[j >> 1][m[j]]));
    }
    st_rlx_d(P.lam + n, lam);
    const unsigned mk = P.mask[n];
    if (mk) {                                              // a reached non-source cell
      P.grad[n] = __dmul_rn(lam, P.grad[n]);
      // no fence here: a cell released now is processed only after the next
      // grid barrier, whose release / acquire publishes every lambda of this level
#pragma unroll
      for (int j = 0; j < 6; ++j) {
        if (!((mk >> j) & 1u)) continue;
        if (atomicSub(P.cnt + m[j], 1) == 1) {
          ready[j] = true;
          ready_entry[j] = entry_of(pi, m[j]);
        }
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 6; ++j) append_ready(count, front, ready[j], ready[j] ? ready_entry[j] : 0ull);
}

__global__ void __launch_bounds__(kThreads) adj_levels_kernel(const AdjProb *probs, int nprob,
                                                               int64_t total, AdjCtl *ctl,
                                                               unsigned long long *front,
                                                               long long timeout_ns) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t warp0 = blockIdx.x * static_cast<int64_t>(blockDim.x) + (threadIdx.x & ~31u);
  const unsigned lane = threadIdx.x & 31u;
  unsigned long long done = 0;
  for (unsigned long long level = 0;; ++level) {
    const int cur = static_cast<int>(level % 3ull);
    const int nxt = static_cast<int>((level + 1ull) % 3ull);
    const unsigned long long n_cur = ld_rlx_u64(&ctl->nfront[cur]);
    if (n_cur == 0) {
      if (blockIdx.x == 0 && threadIdx.x == 0) ctl->levels = level;
      break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->nfront[(level + 2ull) % 3ull] = 0ull;
    const unsigned long long *in = front + (level & 1ull) * static_cast<unsigned long long>(total);
    unsigned long long *out = front + ((level + 1ull) & 1ull) * static_cast<unsigned long long>(total);
    for (int64_t b = warp0; b < static_cast<int64_t>(n_cur); b += stride) {
      const int64_t i = b + lane;
      const bool live = i < static_cast<int64_t>(n_cur);
      adj_process(probs, live ? in[i] : 0ull, live, &ctl->nfront[nxt], out);
      done += live ? 1u : 0u;
    }
    // the other blocks' decrements and lambdas before the next frontier
    if (!grid::barrier(&ctl->bar_count, &ctl->bar_gen, &ctl->status, timeout_ns)) break;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) done += __shfl_xor_sync(kFullMask, done, o);
  if (lane == 0 && done) atomicAdd(&ctl->done, done);
}

// ---------------------------------------------------------------------------
// Tile schedule.  The same per-cell work in the same order as above; the unit
// of scheduling is a tile, given to one warp.  A cell n is ready when every
// downwind user of it (a neighbour m whose mask names n's side) is done.  A visit
// loads the tile and the mask bytes around it: cells with a user across the
// tile edge that is not done are blocked for this visit, the others are
// processed in dependency order, kept as bit sets over the tile (one word per
// lane, as in the forward kernel): ready cells are those none of whose in-tile
// users is left, packed onto the lanes.  Each sums g and the products of its
// users in the fixed order (x-, x+, y-, y+, z-, z+) and turns its weights W_k
// into products p_k = fl(lambda W_k), which is all its upwind cells need.  Then
// the tile's gradients are written, the products that another tile or a later
// visit reads, after a fence the mask bytes with kDone, and the tiles that hold
// upwind cells of this tile's are activated.
//
// The forward solver's bucket scheduler orders the tiles by decreasing time (of
// the cell in the tile's middle, in fractions of the problem's largest time), so
// that a tile's users are mostly done when it is taken.
//
// What bounds it: the chain of tiles.  A visit is 56 kcycles in 2D (32 problems of
// 1024^2 cells: loads 18, 21 rounds 26, stores and hand-over 13; 1.6 visits per tile)
// and 33 in 3D (8 of 90 x 101 x 110: 11, 10 and 12; 3.1 visits), at 4 to 16 % of the
// issue slots, so many small tiles in flight count, and few visits per tile.  Against per-cell counts (two arrays, atomics in the
// set-up and at every release), a FIFO of tiles and a block of 128 (2D) or 256
// threads per tile with a barrier per round: 8.97 -> 4.97 ms for 32 problems of
// 1024^2 cells, 6.6 -> 3.6 ms for one of 192 x 224 x 208.  Tiles: 16x16 in 2D
// (16x8 and 8x8: 9.8 and 10.5 ms against 8.9 for set-up and tiles), 8x4x4 in 3D
// (8x8x4 and 4x4x4: 4.7 and 4.9 against 4.5).  12 warps per SM (20 are slower:
// 10.4 and 6.2 ms; the tiles wait for each other, not for a warp).  Steps of the
// order: 0.04 (nx + ny + nz) per field in 2D (0.25: 11.2 ms, 0.1: 10.2, none:
// 10.1, against 9.8), 0.15 in 3D (0.25: 4.90, 0.04: 4.95, none: 6.3, against 4.85).
// ---------------------------------------------------------------------------
template <int D, int TX, int TY, int TZ>
struct ATile {
  static constexpr int NT = TX * TY * TZ, NC = NT / 32;
  static constexpr int HZ = D == 3 ? 1 : 0;
  static constexpr int SX = TX + 2, SY = TY + 2, SZ = TZ + 2 * HZ, NS = SX * SY * SZ;
  double p[D][NS];                 // W_k, p_k once done (halo: p_k of the axis across the face)
  double lam[NT];                  // g, lambda once done
  unsigned char m[NS];             // mask bytes with halo
  unsigned char list[NT];
};

__device__ __forceinline__ unsigned ld_rlx_u8(const unsigned char *p) {
  unsigned short v;
  asm volatile("ld.relaxed.gpu.global.u8 %0, [%1];" : "=h"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_rlx_u8(unsigned char *p, unsigned v) {
  asm volatile("st.relaxed.gpu.global.u8 [%0], %1;" ::"l"(p), "h"(static_cast<unsigned short>(v)) : "memory");
}

__device__ __forceinline__ int find_tile_prob(const AdjProb *probs, int nprob, unsigned tile) {
  int lo = 0, hi = nprob - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (static_cast<unsigned long long>(ldg_i64(&probs[mid].tile_base)) <= tile) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Bucket of tile (tx, ty, tz) of P: how far its middle cell lies below the
// problem's largest time, in steps of about two cells.
template <int TX, int TY, int TZ>
__device__ __forceinline__ unsigned tile_bucket(const AdjProb &P, unsigned tx, unsigned ty, unsigned tz) {
  const int64_t nx = ldg_i64(&P.nx), ny = ldg_i64(&P.ny), nz = ldg_i64(&P.nz);
  const int64_t mx = static_cast<int64_t>(tx) * TX + TX / 2, my = static_cast<int64_t>(ty) * TY + TY / 2,
                mz = static_cast<int64_t>(tz) * TZ + TZ / 2;
  const int64_t x = mx < nx ? mx : nx - 1, y = my < ny ? my : ny - 1, z = mz < nz ? mz : nz - 1;
  const double *const t = reinterpret_cast<const double *>(ldg_i64(&P.t));
  const unsigned long long tb = static_cast<unsigned long long>(ldg_i64(t + (z * ny + y) * nx + x)),
                           top = static_cast<unsigned long long>(ldg_i64(reinterpret_cast<const void *>(ldg_i64(&P.tmax))));
  const int se = static_cast<int>(top >> 52) - 1023;
  const float f = to_f_scaled(tb, se), ft = to_f_scaled(top, se);
  if (!(f < ft)) return 0u;
  const float steps = (TZ > 1 ? 0.15f : 0.04f) * static_cast<float>(nx + ny + nz);
  return static_cast<unsigned>((ft - f) / ft * fminf(steps, 1.0e6f));
}

// Queue the tiles holding a ready cell: reached, not done, and no neighbour that
// is not done names its side.
template <int TX, int TY, int TZ, bool ROWS>
__global__ void adj_tile_seed_kernel(const AdjProb *probs, int nprob, int64_t total, int first, SolveParams sp) {
  for_cells(probs, nprob, total, first, ROWS, [&](const AdjProb &P, int64_t n) {
    const unsigned char *const mask = P.mask;
    const int64_t sy = P.nx, sz = P.nx * P.ny;
    if ((mask[n] & (kPending | kDone)) != kPending) return;
    const Cell e = cell_of(P, n);
    // neighbour at n + d waits for n, its side `side`
    auto uses = [&](int64_t d, int side) { return ((mask[n + d] >> side) & 1u) && !(mask[n + d] & kDone); };
    const bool used = (e.c[0] > 0 && uses(-1, 1)) || (e.c[0] + 1 < P.nx && uses(1, 0)) ||
                      (e.c[1] > 0 && uses(-sy, 3)) || (e.c[1] + 1 < P.ny && uses(sy, 2)) ||
                      (P.ndim == 3 && ((e.c[2] > 0 && uses(-sz, 5)) || (e.c[2] + 1 < P.nz && uses(sz, 4))));
    if (used) return;
    const unsigned tx = static_cast<unsigned>(e.c[0] / TX), ty = static_cast<unsigned>(e.c[1] / TY),
                   tz = static_cast<unsigned>(e.c[2] / TZ);
    activate(sp, static_cast<unsigned long long>(P.tile_base) + (tz * P.nty + ty) * P.ntx + tx, 0u,
             tile_bucket<TX, TY, TZ>(P, tx, ty, tz));
  }, [](const AdjProb &) {});
}

// TIMING: clocks of the visit phases and of the waits for work (the eik_stats
// timing fields); without it those reads compile out.
template <int D, int TX, int TY, int TZ, bool TIMING>
__global__ void __launch_bounds__(32, kAdjCtas) adj_tiles_kernel(const AdjProb *probs, int nprob, AdjCtl *ctl,
                                                                SolveParams sp) {
  using S = ATile<D, TX, TY, TZ>;
  constexpr int NT = S::NT, NC = S::NC, HZ = S::HZ, SX = S::SX, SY = S::SY;
  static_assert(NT % 32 == 0 && NT <= 256, "whole warps, 8-bit list entries");
  constexpr int kStride[3] = {1, SX, SX * SY};
  constexpr int kTile[3] = {TX, TY, TZ};
  __shared__ S s;
  const int lane = threadIdx.x;
  auto pos_of = [](int q) { return ((q / (TX * TY) + HZ) * SY + (q / TX) % TY + 1) * SX + q % TX + 1; };
  unsigned long long visits = 0, rounds = 0, visit_ns = 0, idle_ns = 0, cyc[4] = {0, 0, 0, 0};
  long long idle_since = 0, t_mark = 0, c0 = 0;
  auto lap = [&](int i) {
    if constexpr (TIMING) {
      const long long c1 = clock64();
      cyc[i] += static_cast<unsigned long long>(c1 - c0);
      c0 = c1;
    }
  };
  if constexpr (TIMING) {
    c0 = clock64();
    t_mark = now_ns();
  }
#pragma unroll 1
  for (;;) {
    long long tile = -1;
    unsigned slot = 0, lo = 0;
#pragma unroll 1
    for (;;) {
      const unsigned long long e = pop_entry(sp, idle_since, slot, lo);
      if (e == kEmpty) break;
      int f = -1;
      if (lane == 0) f = try_claim(sp, e & 0xffffffffull, static_cast<unsigned>(e >> 32));
      f = __shfl_sync(kFull, f, 0);
      if (f >= 0) { tile = static_cast<long long>(e & 0xffffffffull); break; }
      if (lane == 0) {
        atomicAdd(&sp.ctl->run[slot * kCounterPad], 0xffffffffu);
        atomicAdd(&sp.ctl->work, -1);
      }
    }
    if (tile < 0) break;
    idle_since = 0;
    ++visits;
    if constexpr (TIMING) {
      const long long now = now_ns();
      idle_ns += static_cast<unsigned long long>(now - t_mark);
      t_mark = now;
    }
    lap(0);
    // the problem's record through the read-only path: the fence below would
    // send each of these reads to L2
    const AdjProb &P = probs[find_tile_prob(probs, nprob, static_cast<unsigned>(tile))];
    const int64_t nx = ldg_i64(&P.nx), ny = ldg_i64(&P.ny), nz = ldg_i64(&P.nz);
    unsigned tc[3];
    {   // fewer than 2^31 tiles: 32-bit divisions
      const unsigned lt = static_cast<unsigned>(tile - ldg_i64(&P.tile_base)),
                     ntx = static_cast<unsigned>(ldg_i64(&P.ntx)), nty = static_cast<unsigned>(ldg_i64(&P.nty));
      const unsigned rest = lt / ntx;
      tc[0] = lt - rest * ntx;
      tc[2] = rest / nty;
      tc[1] = rest - tc[2] * nty;
    }
    const int64_t x0 = static_cast<int64_t>(tc[0]) * TX, y0 = static_cast<int64_t>(tc[1]) * TY,
                  z0 = static_cast<int64_t>(tc[2]) * TZ;
    const int64_t sy = nx, sz = nx * ny, first = z0 * sz + y0 * sy + x0;
    unsigned char *const mask = reinterpret_cast<unsigned char *>(ldg_i64(&P.mask)) + first;
    double *const grad = reinterpret_cast<double *>(ldg_i64(&P.grad)) + first;
    const double *const gin = reinterpret_cast<const double *>(ldg_i64(&P.g));
    double *W[D];
#pragma unroll
    for (int ax = 0; ax < D; ++ax) W[ax] = reinterpret_cast<double *>(ldg_i64(&P.W[ax])) + first;
    fence_ar();      // the claim is ordered before the tile's loads
    const int xlo = x0 > 0 ? -1 : 0, ylo = y0 > 0 ? -1 : 0, zlo = z0 > 0 ? -1 : 0;
    const int xhi = nx - x0 > TX ? TX + 1 : static_cast<int>(nx - x0);
    const int yhi = ny - y0 > TY ? TY + 1 : static_cast<int>(ny - y0);
    const int zhi = nz - z0 > TZ ? TZ + 1 : static_cast<int>(nz - z0);
    double coef[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const int q = k * 32 + lane, ps = pos_of(q);
      const int ix = q % TX, iy = (q / TX) % TY, iz = q / (TX * TY);
      const bool in = ix < xhi && iy < yhi && iz < zhi;
      const int64_t off = iz * sz + iy * sy + ix;
      s.m[ps] = static_cast<unsigned char>(in ? ld_rlx_u8(mask + off) : 0u);
      coef[k] = in ? grad[off] : 0.0;
      s.lam[q] = in && gin ? gin[first + off] : 0.0;
#pragma unroll
      for (int ax = 0; ax < D; ++ax) s.p[ax][ps] = in ? ld_rlx_d(W[ax] + off) : 0.0;
    }
    constexpr int FX = TY * TZ, FY = TX * TZ, FZ = (D == 3) ? TX * TY : 0;
    constexpr int H = 2 * FX + 2 * FY + 2 * FZ, HC = (H + 31) / 32;
    // halo faces: y (x fastest: coalesced), z, x.  face j of halo cell i
    auto halo = [](int i, int &ix, int &iy, int &iz) -> int {
      if (i < 2 * FY) {
        const int j = i % FY;
        ix = j % TX; iz = j / TX; iy = i < FY ? -1 : TY;
        return i < FY ? 2 : 3;
      }
      if (i < 2 * FY + 2 * FZ) {
        const int k = i - 2 * FY, j = k % (FZ > 0 ? FZ : 1);
        ix = j % TX; iy = j / TX; iz = k < FZ ? -1 : TZ;
        return k < FZ ? 4 : 5;
      }
      const int k = i - 2 * FY - 2 * FZ, j = k % FX;
      iy = j % TY; iz = j / TY; ix = k < FX ? -1 : TX;
      return k < FX ? 0 : 1;
    };
    unsigned hm[HC];
#pragma unroll
    for (int c = 0; c < HC; ++c) {
      const int i = c * 32 + lane;
      int ix, iy, iz;
      halo(i, ix, iy, iz);
      const bool in = i < H && ix >= xlo && ix < xhi && iy >= ylo && iy < yhi && iz >= zlo && iz < zhi;
      hm[c] = in ? ld_rlx_u8(mask + iz * sz + iy * sy + ix) : 0u;
      if (i < H) s.m[((iz + HZ) * SY + iy + 1) * SX + ix + 1] = static_cast<unsigned char>(hm[c]);
    }
    fence_ar();      // a user seen done has its products published
#pragma unroll
    for (int c = 0; c < HC; ++c) {
      const int i = c * 32 + lane;
      int ix, iy, iz;
      const int j = halo(i, ix, iy, iz);
      if (i < H && (hm[c] & kDone) && ((hm[c] >> (j ^ 1)) & 1u))
        s.p[j >> 1][((iz + HZ) * SY + iy + 1) * SX + ix + 1] =
            ld_rlx_d(W[j >> 1] + iz * sz + iy * sy + ix);
    }
    __syncwarp();
    // word k of these sets in lane k: cells to do, cells with a user across the
    // tile edge that is not done, cells with a user in the tile across face j
    unsigned todo_w = 0u, blocked_w = 0u, user_w[2 * D];
#pragma unroll
    for (int j = 0; j < 2 * D; ++j) user_w[j] = 0u;
#pragma unroll 1
    for (int k = 0; k < NC; ++k) {
      const int q = k * 32 + lane, ps = pos_of(q);
      const int cc[3] = {q % TX, (q / TX) % TY, q / (TX * TY)};
      const unsigned own = s.m[ps];
      bool blocked = false;
#pragma unroll
      for (int j = 0; j < 2 * D; ++j) {
        const int ax = j >> 1;
        const unsigned mn = s.m[ps + ((j & 1) ? kStride[ax] : -kStride[ax])];
        const bool user = (mn >> (j ^ 1)) & 1u, inside = cc[ax] != ((j & 1) ? kTile[ax] - 1 : 0);
        blocked = blocked || (user && !inside && !(mn & kDone));
        const unsigned b = __ballot_sync(kFull, user && inside);
        if (lane == k) user_w[j] = b;
      }
      const unsigned bt = __ballot_sync(kFull, (own & kPending) && !(own & kDone));
      const unsigned bb = __ballot_sync(kFull, blocked);
      if (lane == k) { todo_w = bt; blocked_w = bb; }
    }
    const unsigned todo0_w = todo_w;
    lap(1);
#pragma unroll 1
    for (int round = 0; round <= NT; ++round) {
      unsigned ready_w = todo_w & ~blocked_w;
#pragma unroll
      for (int j = 0; j < 2 * D; ++j) ready_w &= ~(user_w[j] & face_bits<TX, TY, TZ>(todo_w, j));
      const int n = list_of_set<NC>(ready_w, s.list);
      __syncwarp();
      if (n == 0) break;
      ++rounds;
      todo_w &= ~ready_w;
#pragma unroll 1
      for (int b = lane; b < n; b += 32) {
        const int q = s.list[b], ps = pos_of(q);
        double lam = s.lam[q];
        const unsigned own = s.m[ps];
#pragma unroll
        for (int j = 0; j < 2 * D; ++j) {
          const int nb = ps + ((j & 1) ? kStride[j >> 1] : -kStride[j >> 1]);
          const unsigned mn = s.m[nb];
          const double pr = s.p[j >> 1][nb];
          if ((mn >> (j ^ 1)) & 1u) lam = __dadd_rn(lam, pr);
        }
#pragma unroll
        for (int ax = 0; ax < D; ++ax)
          if ((own >> (2 * ax)) & 3u) s.p[ax][ps] = __dmul_rn(lam, s.p[ax][ps]);
        s.lam[q] = lam;
      }
      __syncwarp();
    }
    lap(2);
    const unsigned done_w = todo0_w & ~todo_w;
    if (__any_sync(kFull, done_w != 0u)) {
      const bool whole = !__any_sync(kFull, todo_w != 0u);   // no later visit reads this tile's products
      unsigned out_any = 0u, ndone = 0u;
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        const unsigned w = __shfl_sync(kFull, done_w, k);
        ndone += __popc(w);
        if (!((w >> lane) & 1u)) continue;
        const int q = k * 32 + lane, ps = pos_of(q);
        const int cc[3] = {q % TX, (q / TX) % TY, q / (TX * TY)};
        const int64_t off = cc[2] * sz + cc[1] * sy + cc[0];
        const unsigned own = s.m[ps];
        if (own & 0x3fu) grad[off] = __dmul_rn(s.lam[q], coef[k]);
#pragma unroll
        for (int ax = 0; ax < D; ++ax) {
          const bool out_lo = ((own >> (2 * ax)) & 1u) && cc[ax] == 0;
          const bool out_hi = ((own >> (2 * ax + 1)) & 1u) && cc[ax] == kTile[ax] - 1;
          if (out_lo) out_any |= 1u << (2 * ax);
          if (out_hi) out_any |= 1u << (2 * ax + 1);
          if (out_lo || out_hi || (!whole && ((own >> (2 * ax)) & 3u))) st_rlx_d(W[ax] + off, s.p[ax][ps]);
        }
      }
      fence_ar();                               // products before the mask bytes that name them done
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        const unsigned w = __shfl_sync(kFull, done_w, k);
        if (!((w >> lane) & 1u)) continue;
        const int q = k * 32 + lane;
        const int64_t off = (q / (TX * TY)) * sz + ((q / TX) % TY) * sy + q % TX;
        st_rlx_u8(mask + off, s.m[pos_of(q)] | kDone);   // other tiles' visits read it meanwhile
      }
      out_any = __reduce_or_sync(kFull, out_any);
      __syncwarp();
      fence_ar();                               // every lane's stores before the activations
      if ((out_any >> lane) & 1u) {                  // an upwind cell on face j lies in the grid
        const int ax = lane >> 1, d = (lane & 1) ? 1 : -1;
        const unsigned ux = tc[0] + (ax == 0 ? d : 0), uy = tc[1] + (ax == 1 ? d : 0), uz = tc[2] + (ax == 2 ? d : 0);
        activate(sp, static_cast<unsigned long long>(P.tile_base) + (uz * P.nty + uy) * P.ntx + ux, 0u,
                 tile_bucket<TX, TY, TZ>(P, ux, uy, uz), lo);
      }
      __syncwarp();
      if (lane == 0) atomicAdd(&ctl->done, static_cast<unsigned long long>(ndone));
    }
    if (lane == 0) {
      fence_ar();                               // and before the tile is another visit's
      finish_tile(sp, static_cast<unsigned long long>(tile));
      atomicAdd(&sp.ctl->run[slot * kCounterPad], 0xffffffffu);
      atomicAdd(&sp.ctl->work, -1);
    }
    __syncwarp();
    lap(3);
    if constexpr (TIMING) {
      const long long now = now_ns();
      visit_ns += static_cast<unsigned long long>(now - t_mark);
      t_mark = now;
    }
  }
  if (lane == 0) {
    atomicAdd(&ctl->visits, visits);
    atomicAdd(&ctl->rounds, rounds);
    atomicAdd(&ctl->ctas, 1ull);
    if constexpr (TIMING) {
      atomicAdd(&ctl->visit_ns, visit_ns);
      atomicAdd(&ctl->idle_ns, idle_ns);
#pragma unroll
      for (int i = 0; i < 4; ++i) atomicAdd(&ctl->cycles[i], cyc[i]);
    }
  }
}

int g_sms = 0;

int sms() {
  if (!g_sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
    if (g_sms <= 0) g_sms = 1;
  }
  return g_sms;
}

}  // namespace

cudaError_t launch_adjoint(const AdjProb *probs_dev, int nprob, int64_t total, AdjCtl *ctl,
                           unsigned long long *front, long long timeout_ns, cudaStream_t stream) {
  int64_t g = (total + 255) / 256;
  if (g > 8 * sms()) g = 8 * sms();
  if (g < 1) g = 1;
  adj_setup_kernel<<<static_cast<int>(g), 256, 0, stream>>>(probs_dev, nprob, total, ctl);
  adj_seed_kernel<<<static_cast<int>(g), 256, 0, stream>>>(probs_dev, nprob, total, ctl, front);
  note_launches(2);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // co-resident blocks only: the levels meet at a grid barrier
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, adj_levels_kernel, kThreads, 0);
  if (e != cudaSuccess) return e;
  if (per_sm > 2) per_sm = 2;
  if (per_sm < 1) return cudaErrorCooperativeLaunchTooLarge;
#ifndef EIK_ADJ_BLOCK_DIV
#define EIK_ADJ_BLOCK_DIV 4
#endif
  // a quarter of the SMs' worth of 1024-thread blocks: a level rarely holds more
  // ready cells, and fewer, fuller blocks measured faster (32-source 1024^2:
  // 48.8 -> 43.5 ms)
  int blocks = sms() * per_sm / EIK_ADJ_BLOCK_DIV;
  if (blocks < 1) blocks = 1;
  void *args[] = {const_cast<AdjProb **>(&probs_dev), &nprob, &total, &ctl, &front, &timeout_ns};
  e = cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(adj_levels_kernel), dim3(blocks),
                                  dim3(kThreads), args, 0, stream);
  note_launches(1);
  return e;
}

namespace {

template <int D, int TX, int TY, int TZ>
cudaError_t run_tiles(const AdjProb *probs_dev, int nprob, int64_t total, int64_t max_cells, int64_t total_tiles,
                      AdjCtl *ctl, const SolveParams &sp, int ctas_per_sm, bool timing, bool resume, cudaStream_t stream) {
  const int64_t all = static_cast<int64_t>(sms()) * 8, mean = total / nprob;
  auto blocks_for = [](int64_t cells, int64_t most) {
    const int64_t g = (cells + 255) / 256;
    return static_cast<unsigned>(g < 1 ? 1 : g > most ? most : g);
  };
  if (max_cells <= 2 * mean) {
    const unsigned gx = blocks_for(mean, (all + nprob - 1) / nprob);
    for (int step = resume ? 1 : 0; step < 2; ++step) {
      for (int first = 0; first < nprob; first += 65535) {
        const dim3 grid(gx, static_cast<unsigned>(nprob - first < 65535 ? nprob - first : 65535));
        if (step == 0) adj_setup_tiles_kernel<true><<<grid, 256, 0, stream>>>(probs_dev, nprob, total, first, ctl);
        else adj_tile_seed_kernel<TX, TY, TZ, true><<<grid, 256, 0, stream>>>(probs_dev, nprob, total, first, sp);
        note_launches(1);
      }
    }
  } else {
    const unsigned gx = blocks_for(total, all);
    if (!resume) {
      adj_setup_tiles_kernel<false><<<gx, 256, 0, stream>>>(probs_dev, nprob, total, 0, ctl);
      note_launches(1);
    }
    adj_tile_seed_kernel<TX, TY, TZ, false><<<gx, 256, 0, stream>>>(probs_dev, nprob, total, 0, sp);
    note_launches(1);
  }
  // ctas_per_sm 0: what the fronts can use (a front of a problem of n tiles is
  // about n^(1/2) tiles in 2D, n^(2/3) in 3D), since idle warps only hold up the
  // scheduler: 2D 9 problems of 700 x 700 with 2, 4, 8 and 12 per SM 3.28, 3.09, 3.27
  // and 3.66 ms, 4 of 600 x 500 2.05, 2.08, 2.25 and 2.49 ms; 3D one of 100^3 2.65,
  // 2.72, 3.25 and 4.06 ms, 4 of 110 x 90 x 100 4.88, 3.30, 3.01 and 3.33 ms
  int per_sm = D == 3 ? 10 : kAdjCtas;
  if (ctas_per_sm > 0) {
    per_sm = ctas_per_sm < kAdjCtas ? ctas_per_sm : kAdjCtas;
  } else {
    const double each = static_cast<double>(total_tiles) / nprob;
    const double want = nprob * (D == 3 ? 0.75 * cbrt(each) * cbrt(each) : 1.5 * sqrt(each)) / sms();
    if (want < per_sm) per_sm = want > 2.0 ? static_cast<int>(ceil(want)) : 2;
  }
  int64_t blocks = static_cast<int64_t>(sms()) * per_sm;
  if (blocks > total_tiles) blocks = total_tiles;
  if (blocks < 1) blocks = 1;
  if (timing)
    adj_tiles_kernel<D, TX, TY, TZ, true><<<static_cast<int>(blocks), 32, 0, stream>>>(probs_dev, nprob, ctl, sp);
  else
    adj_tiles_kernel<D, TX, TY, TZ, false><<<static_cast<int>(blocks), 32, 0, stream>>>(probs_dev, nprob, ctl, sp);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_adj_h2s(const double *v, int v_is_slowness, double hh, int64_t n, double *hs,
                           cudaStream_t stream) {
  int64_t g = (n + 255) / 256;
  if (g > 8 * sms()) g = 8 * sms();
  adj_h2s_kernel<<<static_cast<int>(g < 1 ? 1 : g), 256, 0, stream>>>(v, v_is_slowness, hh, n, hs);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_tiles(const AdjProb *probs_dev, int nprob, int64_t total, int64_t max_cells,
                                 int64_t total_tiles, int ndim, AdjCtl *ctl, const SolveParams &sp, int ctas_per_sm,
                                 bool timing, bool resume, cudaStream_t stream) {
  if (ndim == 3)
    return run_tiles<3, kAdjTile3[0], kAdjTile3[1], kAdjTile3[2]>(probs_dev, nprob, total, max_cells, total_tiles, ctl,
                                                                  sp, ctas_per_sm, timing, resume, stream);
  return run_tiles<2, kAdjTile2[0], kAdjTile2[1], kAdjTile2[2]>(probs_dev, nprob, total, max_cells, total_tiles, ctl,
                                                                sp, ctas_per_sm, timing, resume, stream);
}

}  // namespace eik
