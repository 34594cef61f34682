// Window search: the search of sas_stack (Sec. 2.1 steps 1-3) in two levels.
//
// The one-level stack kernel adds every (detection, velocity) pair to a counter.
// Nearly all of those counters stay far below N_min.  Here the lattice is first
// searched in groups of gx x gy velocities:
//
//   Level 1 projects each detection with the group's centre velocity V only and
//   counts it in a grid of square cells of P mpx (k_stack in window mode, sas_
//   stack_windows.cu).  A detection of the bin with lower corner p at velocity v
//   of the group projects at V to u = p + (s_v - S_V) + (0 .. bin - 1), and over
//   the epochs s_v - S_V runs from m(v) to M(v).  So all detections of that bin
//   lie in [p + m, p + M + bin - 1]: no longer than (win - 1) P + 1 by the
//   choice of P, hence inside the window of win x win cells that begins in the
//   cell of p + m.  The windows whose sum reaches N_min therefore hold every bin
//   that does, and each (velocity, bin) belongs to one window.
//
//   Level 2 (k_window_cells, a warp per such window) lists the window's
//   detections once and counts, for all velocities of the group at a time, the
//   bins that belong to the window; where a raw count reaches N_min it counts the
//   distinct epochs exactly, from the list, and appends the candidate's key.
//
// The number of (detection, velocity) pairs in the domain, which the result
// reports, is counted directly: per axis the lattice points that keep a
// detection inside form a range (the shift is monotone in the lattice index), so
// a detection's pairs are a rectangle of the lattice (k_window_pairs).
//
// plan_windows picks the group, the window side and the cell from the expected
// instructions of both levels, and leaves the search to the one-level kernel
// where the noise alone would fill the windows.  At 2048 x 4096 px, 100 epochs and
// 12,321 velocities level 1 takes 145 us and level 2 235 us, where the one-level
// kernel and its exact counts took 1360 + 270 us; with a million velocities 8.9 ms
// and 0.32 ms instead of 71.4 ms.  Level 1 is bound by shared memory and barriers
// (58 % of the shared pipe, 48 % of the issue slots).  Everything stays exact whatever
// the choice.  A window of more detections than a warp lists at first is counted by a
// second pass with longer lists, a window list that overflows is made longer, and 8-bit
// counters that wrap are replaced by 16-bit ones; a 16-bit counter that wraps or a window of
// more than the longer lists hold makes the host run the one-level search instead.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdlib>

#include "sas_count.cuh"

namespace sas {

namespace {

constexpr int kWarps = 8;         // warps of a level-2 block
constexpr uint32_t kList = 256, kLongList = 2048;  // detections a warp's list holds: at first, and of a long window
constexpr int kMaxOwn = 2;        // bins per axis that a window owns at one velocity (P <= 2 bins)
constexpr int kMaxWindowEpochs = 255;

__device__ __forceinline__ bool searched(const SearchGeom& g, int kx, int ky) {
  if (kx >= g.nvx || ky >= g.nvy) return false;
  const uint64_t v = (uint64_t)ky * g.nvx + kx;
  if (v < g.v_begin || v >= g.v_end) return false;
  if (g.smin == 0 && g.smax == 0) return true;
  const int64_t vx = (int64_t)g.vx0 + (int64_t)kx * g.dvx, vy = (int64_t)g.vy0 + (int64_t)ky * g.dvy;
  const int64_t s2 = vx * vx + vy * vy;
  return s2 >= (int64_t)g.smin * g.smin && s2 <= (int64_t)g.smax * g.smax;
}

// One warp per fine lattice column, then per row: the group centre's shifts and
// the least difference of the fine ones from them.
__global__ void __launch_bounds__(kWarps * 32) k_window_tables(WindowArgs a) {
  const int w = blockIdx.x * kWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const bool y_axis = w >= a.g.nvx;
  const int k = y_axis ? w - a.g.nvx : w;
  if (y_axis && k >= a.g.nvy) return;
  const int grp = y_axis ? a.gy : a.gx, K = k / grp;
  const uint32_t E = a.g.E;
  const int64_t v2 = 2 * (int64_t)(y_axis ? a.g.vy0 : a.g.vx0) +
                     (int64_t)(2 * K * grp + grp - 1) * (y_axis ? a.g.dvy : a.g.dvx);
  const int32_t* fine = (y_axis ? a.syt : a.sxt) + (size_t)k * E;
  int32_t* centre = (y_axis ? a.sYt : a.sXt) + (size_t)K * E;
  int32_t lo = INT32_MAX, hi = INT32_MIN;
  for (uint32_t e = lane; e < E; e += 32) {
    const int64_t s64 = floor_div64(v2 * a.dt[e], 2 * a.g.tph);
    const int32_t S = s64 > -kLimDomain && s64 < kLimDomain ? (int32_t)s64 : 0;
    if (k % grp == 0) centre[e] = S;
    if (a.ecount[e] > 0) {
      lo = min(lo, fine[e] - S);
      hi = max(hi, fine[e] - S);
    }
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) {
    (y_axis ? a.my : a.mx)[k] = lo;
    // the bin's detections fit the window, and its corner lies on the grid of cells
    const int64_t span = (int64_t)a.unit + hi - lo;
    const int64_t margin = y_axis ? (int64_t)a.g.y_min - a.cgm.y_min : (int64_t)a.g.x_min - a.cgm.x_min;
    if (span > (int64_t)(a.win - 1) * a.cgm.bin + 1 || -(int64_t)lo > margin || (int64_t)hi > margin)
      atomicOr(a.flags, kFlagWindow);
  }
}

// Coarse lattice points with a searched fine one: a warp each.
__global__ void __launch_bounds__(kWarps * 32) k_window_active(WindowArgs a) {
  const int i = blockIdx.x * kWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= a.cgm.nvx * a.cgm.nvy) return;
  const int Kx = i % a.cgm.nvx, Ky = i / a.cgm.nvx;
  bool any = false;
  for (int j = lane; j < a.gx * a.gy; j += 32) any |= searched(a.g, Kx * a.gx + j % a.gx, Ky * a.gy + j / a.gx);
  any = __any_sync(0xffffffffu, any);
  if (lane == 0) a.vact[i] = any;
}

// vsum[ky][kx]: searched lattice points with indices below (kx, ky) on both
// axes.  First pass: a warp per row; second: a warp per column.
__global__ void __launch_bounds__(kWarps * 32) k_window_rowsum(WindowArgs a) {
  const int ky = blockIdx.x * kWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (ky > a.g.nvy) return;
  uint32_t* out = a.vsum + (size_t)ky * (a.g.nvx + 1);
  uint32_t run = 0;
  for (int k0 = 0; k0 <= a.g.nvx; k0 += 32) {
    const int kx = k0 + lane;  // out[kx] = row ky - 1's points below kx
    const bool s = ky > 0 && kx < a.g.nvx && searched(a.g, kx, ky - 1);
    const uint32_t m = __ballot_sync(0xffffffffu, s);
    if (kx <= a.g.nvx) out[kx] = run + (uint32_t)__popc(m & ((1u << lane) - 1u));
    run += (uint32_t)__popc(m);
  }
}
__global__ void __launch_bounds__(kWarps * 32) k_window_colsum(WindowArgs a) {
  const int kx = blockIdx.x * kWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (kx > a.g.nvx) return;
  uint32_t run = 0;
  for (int k0 = 0; k0 <= a.g.nvy; k0 += 32) {
    const int ky = k0 + lane;
    uint32_t* p = a.vsum + (size_t)ky * (a.g.nvx + 1) + kx;
    uint32_t v = ky <= a.g.nvy ? *p : 0u;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += t;
    }
    if (ky <= a.g.nvy) *p = run + v;
    run += __shfl_sync(0xffffffffu, v, 31);
  }
}

// First lattice index whose shift reaches a (up: s >= a; else s <= a): the shifts
// t[k * E], k < n, are monotone and within one of a straight line, so a guess
// on that line is off by a step or two; a slope below one mpx a step repeats
// values and is searched by halves.
__device__ __forceinline__ int first_index(const int32_t* __restrict__ t, uint32_t E, int n, int32_t t0, float slope,
                                           bool up, int64_t a) {
  int lo = 0, hi = n;
  if (fabsf(slope) >= 1.f) {
    lo = (int)fminf(fmaxf(((float)(a - t0)) / slope, 0.f), (float)n);
    while (lo > 0 && (up ? t[(size_t)(lo - 1) * E] >= a : t[(size_t)(lo - 1) * E] <= a)) --lo;
    while (lo < n && (up ? t[(size_t)lo * E] < a : t[(size_t)lo * E] > a)) ++lo;
    return lo;
  }
  while (lo < hi) {
    const int m = (lo + hi) >> 1;
    if (up ? t[(size_t)m * E] >= a : t[(size_t)m * E] <= a) hi = m; else lo = m + 1;
  }
  return lo;
}

// Lattice indices [first, last) whose shift keeps coordinate x (relative to the
// domain's edge) inside [0, width).
__device__ __forceinline__ void inside_range(const int32_t* __restrict__ t, uint32_t E, int n, int64_t x, int64_t width,
                                             int& first, int& last) {
  const int32_t t0 = t[0], t1 = t[(size_t)(n - 1) * E];
  const bool up = t1 >= t0;
  const float slope = n > 1 ? ((float)t1 - (float)t0) / (float)(n - 1) : 0.f;
  first = first_index(t, E, n, t0, slope, up, up ? x - width + 1 : x);
  last = max(first, first_index(t, E, n, t0, slope, up, up ? x + 1 : x - width));
}

__global__ void __launch_bounds__(256) k_window_pairs(WindowArgs a, const int32_t* __restrict__ x,
                                                      const int32_t* __restrict__ y,
                                                      const uint16_t* __restrict__ epoch, uint64_t n) {
  unsigned long long sum = 0;
  const SearchGeom& g = a.g;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t e = epoch[i];
    if (e >= g.E) continue;  // reported by the ingest
    int xa, xb, ya, yb;
    inside_range(a.sxt + e, g.E, g.nvx, (int64_t)x[i] - g.x_min, (int64_t)g.nbx * g.bin, xa, xb);
    inside_range(a.syt + e, g.E, g.nvy, (int64_t)y[i] - g.y_min, (int64_t)g.nby * g.bin, ya, yb);
    if (xa >= xb || ya >= yb) continue;
    if (!a.vsum) {
      sum += (unsigned long long)(xb - xa) * (unsigned long long)(yb - ya);
    } else {
      const size_t r = g.nvx + 1;
      sum += (a.vsum[yb * r + xb] - a.vsum[yb * r + xa]) - (a.vsum[ya * r + xb] - a.vsum[ya * r + xa]);
    }
  }
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if ((threadIdx.x & 31) == 0 && sum) atomicAdd(a.n_pairs, sum);
}

// ---- level 2 ------------------------------------------------------------------

// A warp's window: its detections relative to the window's corner.
template <bool W, uint32_t N>
struct WarpList {
  int32_t x[N], y[N];
  uint8_t e[N];
  uint8_t w[W ? N : 4];           // weights
  uint32_t seen[W ? 256 : 8];     // of the bin being counted: its epochs' bits, or their largest weights
  // per lattice column (8) and row (8) of the group: first owned bin, offset of its
  // edge, and the lengths of the first and second owned bin (0: not owned)
  int32_t first[16], off[16], len0[16], len1[16];
};

// The runs of bucketed detections under a window at an epoch: at most two bucket
// rows (a bucket is no smaller than a window), and the window's corner there.
struct Runs {
  uint32_t k, k1, j, j1;
  int32_t ox, oy;
};
__device__ __forceinline__ Runs window_runs(const WindowArgs& a, const int32_t* SX, const int32_t* SY, uint32_t e,
                                            int32_t ux0, int32_t uy0, int span, uint64_t cell_m) {
  Runs r{};
  if (e >= a.g.E || a.ecount[e] == 0) return r;
  const CoarseGeom& cg = a.cg;
  r.ox = ux0 + SX[e];
  r.oy = uy0 + SY[e];
  int cxa, cxb, cya, cyb;
  bucket_range(r.ox - cg.gx0, span, cell_m, cg.ncx, cxa, cxb);
  bucket_range(r.oy - cg.gy0, span, cell_m, cg.ncy, cya, cyb);
  if (cxa > cxb || cya > cyb) return r;
  const uint32_t* row = a.boff + ((size_t)e * cg.ncy + cya) * cg.ncx;
  r.k = row[cxa];
  r.k1 = row[cxb + 1];
  if (cyb > cya) {
    row += cg.ncx;
    r.j = row[cxa];
    r.j1 = row[cxb + 1];
  }
  return r;
}

constexpr int32_t kOutside = INT32_MIN / 2;  // in no bin, whatever a group's edge adds

// W: weighted stacking.  A bin's sum of weights takes the place of its raw count
// (the masks are counted once per bit of the weights), and the sum of its
// epochs' largest weights that of its distinct epochs.
//
// What bounds it: instruction issue (65 % of the slots at 2048 x 4096 px, 100 epochs,
// 12,321 velocities) and the latency of each window's chain of loads.  Four blocks
// of eight warps an SM; five left fewer registers and were no faster.  Windows
// drawn one by one in a block, records and offsets asked for one turn ahead: 292 ->
// 235 us there, 528 -> 400 us with weights, 380 -> 320 us for a million velocities.
// (Two records a turn cost more instructions than it hid: 277 us, and 107 -> 128 us
// where runs are short.)
//
// LONG: the windows in the queue, with room for kLongList detections each.  A window
// of more than kList (two steady sources in it over 130 epochs, say) is marked by the
// first pass and counted here; fields without such windows do not launch it.  Longer
// lists for all would cost the first pass its occupancy; these leave one block of
// eight warps an SM (163 KB, weighted 174), and a few windows are bound by one warp's
// exact counts, bin after bin: 0.3 ms for one pair of sources at 2048 x 4096 px, 130
// epochs and 12,321 velocities, where the one-level search instead took 5.4 ms more.
template <bool W, bool LONG>
__global__ void __launch_bounds__(kWarps * 32, LONG ? 1 : 4) k_window_cells(WindowArgs a, uint64_t cell_m) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31;
  constexpr uint32_t kCap = LONG ? kLongList : kList;
  using List = WarpList<W, kCap>;
  List& L = reinterpret_cast<List*>(smem)[threadIdx.x >> 5];
  const uint32_t lt = (1u << lane) - 1u;
  const SearchGeom& g = a.g;
  const uint32_t E = g.E;
  const int P = a.cgm.bin, span = a.win * P, nvg = a.gx * a.gy;
  const uint32_t n_win = LONG ? a.n_queue : *a.n_windows;
  const unsigned long long wrapped = LONG ? 0 : *a.balance;  // both loads at once
  if (!LONG && (n_win > a.list_cap || wrapped)) return;  // level 1 runs again: longer list, wider counters
  unsigned long long raw_sum = 0;
  constexpr int kSeen = W ? 256 : 8;
  for (int i = lane; i < kSeen; i += 32) L.seen[i] = 0;
  // sides of a group are powers of two
  const int lgx = __ffs(a.gx) - 1, jx = lane & (a.gx - 1);
  const int jy0 = min(lane >> lgx, a.gy - 1), jy1 = min((lane + 32) >> lgx, a.gy - 1);
  // A block takes every gridDim.x-th row of kWarps windows; its warps draw them one by
  // one, as windows on a mover's track cost several times the others.
  __shared__ uint32_t drawn;
  if (threadIdx.x == 0) drawn = kWarps;
  __syncthreads();
  uint32_t i_win = threadIdx.x >> 5, ahead = 0;
  for (;; i_win = __shfl_sync(0xffffffffu, ahead, 0)) {
    const uint64_t w = ((uint64_t)(i_win / kWarps) * gridDim.x + blockIdx.x) * kWarps + i_win % kWarps;
    if (w >= n_win) break;
    if (lane == 0) ahead = atomicAdd(&drawn, 1u);
    const Emit em = a.windows[LONG ? a.queue[w] : (uint32_t)w];
    const int Kx = (int)(em.v_idx % (uint32_t)a.cgm.nvx), Ky = (int)(em.v_idx / (uint32_t)a.cgm.nvx);
    const int32_t ux0 = a.cgm.x_min + (int32_t)em.bx * P, uy0 = a.cgm.y_min + (int32_t)em.by * P;
    __syncwarp();
    if (lane < 16) {  // the bins that begin in the window's first cell, per column and row of the group
      const bool ya = lane >= 8;
      const int j = lane & 7, grp = ya ? a.gy : a.gx, k = (ya ? Ky : Kx) * grp + j;
      int32_t first = 0, own = 0, off = 0;
      if (j < grp && k < (ya ? g.nvy : g.nvx)) {
        const int32_t rel = (ya ? uy0 - g.y_min : ux0 - g.x_min) - (ya ? a.my : a.mx)[k];
        first = max(-floor_div32(-rel, a.unit), 0);
        own = max(min(floor_div32(rel + P - 1, a.unit), (ya ? g.nby : g.nbx) - 1) - first + 1, 0);
        off = (ya ? uy0 - g.y_min : ux0 - g.x_min) - first * a.unit;
        if (own > kMaxOwn) {  // not by plan_windows' choice of the cell
          atomicOr(a.flags, kFlagWindow);
          own = 0;
        }
      }
      L.first[lane] = first;
      L.off[lane] = off;
      L.len0[lane] = own > 0 ? a.unit : 0;
      L.len1[lane] = own > 1 ? a.unit : 0;
    }
    // The window's detections, a lane per epoch.  The chain of loads (shift, bucket
    // offsets, records) is what a window waits for, so the next 32 epochs' offsets
    // are asked for before these ones' records are walked, and each record before the
    // one ahead of it is looked at.
    const int32_t* SX = a.sXt + (size_t)Kx * E;
    const int32_t* SY = a.sYt + (size_t)Ky * E;
    Runs next = window_runs(a, SX, SY, lane, ux0, uy0, span, cell_m);
    uint32_t n = 0;
    for (uint32_t eb = 0; eb < E; eb += 32) {
      const uint32_t e = eb + lane;
      const Runs r = next;
      if (eb + 32 < E) next = window_runs(a, SX, SY, e + 32, ux0, uy0, span, cell_m);
      const uint32_t na = r.k1 - r.k, total = na + (r.j1 - r.j);
      const int4* ra = reinterpret_cast<const int4*>(a.dets) + r.k;
      const int4* rb = reinterpret_cast<const int4*>(a.dets) + r.j - na;
      const uint32_t most = __reduce_max_sync(0xffffffffu, total);
      int4 ahead_d{};
      if (total > 0) ahead_d = *(na > 0 ? ra : rb);
      for (uint32_t q = 0; q < most; ++q) {
        const int4 d = ahead_d;
        if (q + 1 < total) ahead_d = (q + 1 < na ? ra : rb)[q + 1];
        const int32_t X = d.x - r.ox, Y = d.y - r.oy;
        const bool hit = q < total && (uint32_t)X < (uint32_t)span && (uint32_t)Y < (uint32_t)span;
        const uint32_t m = __ballot_sync(0xffffffffu, hit);
        const uint32_t p = n + (uint32_t)__popc(m & lt);
        if (hit && p < kCap) {
          L.x[p] = X;
          L.y[p] = Y;
          L.e[p] = (uint8_t)e;
          if constexpr (W) L.w[p] = a.wts[(uint32_t)d.w];
        }
        n += (uint32_t)__popc(m);
      }
    }
    if (!W && n < a.n_min) continue;  // warp-uniform (the window's counters also hold the halo's rounding)
    if (n > kCap) {
      if (lane == 0) {
        if constexpr (LONG) {
          atomicOr(a.flags, kFlagWindow);
        } else {
          a.windows[w].flags = kEmitLong;
          atomicAdd(a.n_long, 1u);
        }
      }
      continue;
    }
    __syncwarp();
    // Raw counts of the bins of this lane's velocities (lane and lane + 32 of the
    // group), 32 detections at a time: bit masks over the detections say which lie
    // in each owned bin column at each lattice column and each owned bin row at each
    // lattice row (lane 2 j + c keeps column c's at lattice column j, lane 16 + 2 j + r
    // row r's at lattice row j); a bin's count is the number of bits that its column's
    // and its row's mask share.  Some 250 instructions per 32 detections for up to 256
    // bins, where counting the detections one by one into packed counters took 1100.
    uint32_t raw[2][kMaxOwn][kMaxOwn] = {};
    for (uint32_t i0 = 0; i0 < n; i0 += 32) {
      const uint32_t i = i0 + lane;
      const uint32_t e = i < n ? L.e[i] : 0;
      const int32_t xs = i < n ? L.x[i] + SX[e] : 0, ys = i < n ? L.y[i] + SY[e] : 0;
      const int32_t* sx = a.sxt + (size_t)(Kx * a.gx) * E + e;
      const int32_t* sy = a.syt + (size_t)(Ky * a.gy) * E + e;
      const int cols = i < n ? min(a.gx, g.nvx - Kx * a.gx) : 0, rows = i < n ? min(a.gy, g.nvy - Ky * a.gy) : 0;
      int32_t tx[8], ty[8];  // all loads first, whatever the group's sides
#pragma unroll
      for (int j = 0; j < 8; ++j) tx[j] = j < cols ? xs - sx[(size_t)j * E] : kOutside;
#pragma unroll
      for (int j = 0; j < 8; ++j) ty[j] = j < rows ? ys - sy[(size_t)j * E] : kOutside;
      uint32_t mine = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (j >= a.gx) break;
        const int32_t t = tx[j] + L.off[j];
        const uint32_t m0 = __ballot_sync(0xffffffffu, (uint32_t)t < (uint32_t)L.len0[j]);
        const uint32_t m1 = __ballot_sync(0xffffffffu, (uint32_t)(t - a.unit) < (uint32_t)L.len1[j]);
        if (lane >> 1 == j) mine = lane & 1 ? m1 : m0;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (j >= a.gy) break;
        const int32_t t = ty[j] + L.off[8 + j];
        const uint32_t m0 = __ballot_sync(0xffffffffu, (uint32_t)t < (uint32_t)L.len0[8 + j]);
        const uint32_t m1 = __ballot_sync(0xffffffffu, (uint32_t)(t - a.unit) < (uint32_t)L.len1[8 + j]);
        if (lane >> 1 == 8 + j) mine = lane & 1 ? m1 : m0;
      }
      uint32_t both[2][kMaxOwn][kMaxOwn];
#pragma unroll
      for (int c = 0; c < kMaxOwn; ++c) {
        const uint32_t mc = __shfl_sync(0xffffffffu, mine, 2 * jx + c);
#pragma unroll
        for (int r = 0; r < kMaxOwn; ++r) {
          both[0][r][c] = mc & __shfl_sync(0xffffffffu, mine, 16 + 2 * jy0 + r);
          both[1][r][c] = mc & __shfl_sync(0xffffffffu, mine, 16 + 2 * jy1 + r);
        }
      }
      const uint32_t wi = W && i < n ? L.w[i] : 0u;
#pragma unroll
      for (int b = 0; b < (W ? 8 : 1); ++b) {
        const uint32_t bits = W ? __ballot_sync(0xffffffffu, (wi >> b) & 1u) : 0xffffffffu;
#pragma unroll
        for (int q = 0; q < 2 * kMaxOwn * kMaxOwn; ++q)
          (&raw[0][0][0])[q] += (uint32_t)__popc((&both[0][0][0])[q] & bits) << b;
      }
    }
    // bins whose raw count reaches n_min: bit 4 i + 2 r + c
    uint32_t todo = 0;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int v = lane + 32 * i;
      if (v >= nvg) continue;
      uint32_t t = 0;
#pragma unroll
      for (int r = 0; r < kMaxOwn; ++r)
#pragma unroll
        for (int c = 0; c < kMaxOwn; ++c) t |= (uint32_t)(raw[i][r][c] >= a.n_min) << (2 * r + c);
      if (t && searched(g, Kx * a.gx + jx, Ky * a.gy + (i ? jy1 : jy0))) todo |= t << (4 * i);
    }
    uint32_t who;
    while ((who = __ballot_sync(0xffffffffu, todo != 0)) != 0) {
      const int src = __ffs(who) - 1;
      const int b = __ffs(__shfl_sync(0xffffffffu, todo, src)) - 1;
      if (lane == src) todo &= todo - 1;
      const int v = src + (b & 4 ? 32 : 0), c = b & 1, r = (b >> 1) & 1;
      const int kx = v & (a.gx - 1), ky = v >> lgx;
      const int32_t* sx = a.sxt + (size_t)(Kx * a.gx + kx) * E;
      const int32_t* sy = a.syt + (size_t)(Ky * a.gy + ky) * E;
      const int32_t ax = L.off[kx] - c * a.unit, ay = L.off[8 + ky] - r * a.unit;
      uint32_t raw_n = 0, distinct = 0;
      for (uint32_t i0 = 0; i0 < n; i0 += 32) {
        const uint32_t i = i0 + lane;
        bool in = false, fresh = false;
        if (i < n) {
          const uint32_t e = L.e[i];
          in = (uint32_t)(L.x[i] + SX[e] - sx[e] + ax) < (uint32_t)a.unit &&
               (uint32_t)(L.y[i] + SY[e] - sy[e] + ay) < (uint32_t)a.unit;
          if (in) {
            if constexpr (W) {
              atomicMax(&L.seen[e], (uint32_t)L.w[i]);
            } else {
              const uint32_t bit = 1u << (e & 31);
              fresh = !(atomicOr(&L.seen[e >> 5], bit) & bit);
            }
          }
        }
        raw_n += (uint32_t)__popc(__ballot_sync(0xffffffffu, in));
        distinct += (uint32_t)__popc(__ballot_sync(0xffffffffu, fresh));
      }
      __syncwarp();
      for (int i = lane; i < kSeen; i += 32) {
        if constexpr (W) distinct += L.seen[i];
        L.seen[i] = 0;
      }
      if constexpr (W) distinct = __reduce_add_sync(0xffffffffu, distinct);
      __syncwarp();
      if (distinct >= a.n_min && lane == 0) {
        Key key;
        key.a = ((uint64_t)(~distinct) << 32) | (uint64_t)(~raw_n);
        key.b = ((uint64_t)((uint32_t)(Ky * a.gy + ky) * (uint32_t)g.nvx + (uint32_t)(Kx * a.gx + kx)) << 32) |
                (uint64_t)(uint32_t)(L.first[8 + ky] + r);
        key.c = (uint32_t)(L.first[kx] + c);
        key.pad = 0;
        const uint32_t p = atomicAdd(a.n_valid, 1u);
        if (p < a.key_cap) a.keys[p] = key;
        raw_sum += raw_n;
      }
    }
  }
  if (lane == 0 && raw_sum) atomicAdd(a.raw_total, raw_sum);
}

// Places of the marked windows.
__global__ void __launch_bounds__(1024) k_window_queue(WindowArgs a) {
  const uint32_t n_win = *a.n_windows;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_win; i += gridDim.x * blockDim.x) {
    if (a.windows[i].flags != kEmitLong) continue;
    const uint32_t p = atomicAdd(a.n_long, 1u);
    if (p < a.n_queue) a.queue[p] = i;
  }
}

}  // namespace

cudaError_t launch_window_tables(const WindowArgs& a, cudaStream_t s) {
  k_window_tables<<<(a.g.nvx + a.g.nvy + kWarps - 1) / kWarps, kWarps * 32, 0, s>>>(a);
  note_launch();
  if (a.vact) {
    k_window_active<<<(a.cgm.nvx * a.cgm.nvy + kWarps - 1) / kWarps, kWarps * 32, 0, s>>>(a);
    k_window_rowsum<<<(a.g.nvy + kWarps) / kWarps, kWarps * 32, 0, s>>>(a);
    k_window_colsum<<<(a.g.nvx + kWarps) / kWarps, kWarps * 32, 0, s>>>(a);
    note_launch(3);
  }
  return cudaGetLastError();
}

cudaError_t launch_window_pairs(const WindowArgs& a, const int32_t* x, const int32_t* y, const uint16_t* epoch,
                                uint64_t n, cudaStream_t s) {
  k_window_pairs<<<(unsigned)std::min<uint64_t>((n + 255) / 256, 152 * 8), 256, 0, s>>>(a, x, y, epoch, n);
  note_launch();
  return cudaGetLastError();
}

template <bool W, bool LONG>
static cudaError_t launch_cells(const WindowArgs& a, int blocks, cudaStream_t s) {
  constexpr size_t smem = kWarps * sizeof(WarpList<W, LONG ? kLongList : kList>);
  static_assert(smem <= (LONG ? 225 : 56) * 1024, "one block an SM, or four");
  cudaError_t e = cudaFuncSetAttribute(k_window_cells<W, LONG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_window_cells<W, LONG><<<blocks, kWarps * 32, smem, s>>>(a, div_magic((uint32_t)a.cg.cell));
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_window_cells(const WindowArgs& a, int sms, cudaStream_t s) {
  return a.wts ? launch_cells<true, false>(a, 4 * sms, s) : launch_cells<false, false>(a, 4 * sms, s);
}

cudaError_t launch_window_queue(const WindowArgs& a, int sms, cudaStream_t s) {
  k_window_queue<<<2 * sms, 1024, 0, s>>>(a);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_window_long(const WindowArgs& a, int sms, cudaStream_t s) {
  const int blocks = (int)std::min<uint32_t>((a.n_queue + kWarps - 1) / kWarps, (uint32_t)sms);
  return a.wts ? launch_cells<true, true>(a, blocks, s) : launch_cells<false, true>(a, blocks, s);
}

// ---- planning -----------------------------------------------------------------

void fill_window_args(const WindowPlan& wp, uint32_t n_min, uint32_t ky_lo, uint32_t ky_hi, StackArgs* sa) {
  const TileCfg& tc = wp.tc;
  sa->g = wp.g;
  sa->cg = wp.cg;
  sa->tc = tc;
  sa->win = wp.win;
  sa->magic = magic_for(wp.g.bin);
  sa->bin_is_one = 0;
  sa->merge = 0;
  sa->cell_m = div_magic((uint32_t)wp.cg.cell);
  sa->rows_m = ((1u << 20) + (uint32_t)tc.rows - 1) / (uint32_t)tc.rows;
  sa->n_min = sa->n_low = n_min;
  sa->select = kSelectAll;
  sa->kx_lo = 0;
  sa->ky_lo = (int)ky_lo / wp.gy;
  const uint32_t rows = ky_hi / (uint32_t)wp.gy - (uint32_t)sa->ky_lo + 1;
  sa->nvt_x = (int)div_ceil_u32((uint32_t)wp.g.nvx, (uint32_t)(tc.kx * tc.bvx));
  sa->nvt_y = (int)div_ceil_u32(rows, (uint32_t)(tc.ky * tc.bvy));
  sa->nst_x = (int)div_ceil_u32((uint32_t)wp.g.nbx, (uint32_t)(tc.tx - (wp.win - 1)));
  sa->nst_y = (int)div_ceil_u32((uint32_t)wp.g.nby, (uint32_t)(tc.ty - (wp.win - 1)));
  sa->n_tiles = (uint64_t)sa->nvt_x * sa->nvt_y * sa->nst_x * sa->nst_y;
}

namespace {

// Tile of a window search: the side of its square of cells by the expected cycles
// (returned; 0: none fits), and the bucket cell: as many bucket rows per unit as
// its segments allow (one per epoch and row), since small buckets mean few
// detections that miss the tile or the window.  Cycles: an SM runs
// ceil(units / SMs) units; one takes about 9000 for set-up and barriers, 0.85 per
// cell of 16 lattice points (60 instructions per four words) and 2.5 per candidate
// record (175 instructions per 32), at 2.2 instructions a cycle -- fitted to a
// million-velocity search with its phases left out in turn.
double window_tiles(const sas_grid_desc& d, uint64_t n, uint64_t Ky_lo, uint64_t Ky_hi, double hour, int cb,
                    const DevInfo& di, const FieldPlan& fp, WindowPlan* wp) {
  const uint32_t E = fp.g.E;
  const SearchGeom& g = wp->g;
  TileCfg tc{};
  tc.kx = tc.ky = 4;
  tc.bvx = tc.bvy = 1;
  tc.s = 1;
  tc.cb = cb;
  tc.nt = tc.seg_cap = 1024;
  tc.ec = (int)E;
  tc.emit_cap = 512;
  const int64_t budget = (int64_t)di.smem_optin - 1024;  // room for static shared memory
  const int halo = wp->win - 1;
  const double per_px2 = (double)n / ((double)d.nbx * d.bin * ((double)d.nby * d.bin));
  const double sx = 3.0 * std::fabs((double)g.dvx) * hour + 2.0, sy = 3.0 * std::fabs((double)g.dvy) * hour + 2.0;
  const double vtiles = (double)div_ceil_u32((uint32_t)g.nvx, 4) * (double)div_ceil_u32((uint32_t)(Ky_hi - Ky_lo + 1), 4);
  const int rows = tc.seg_cap / (int)E;  // >= 4
  double best = 0;
  for (int side = 16; side <= 160; side += side / 16 * 4) {
    // even tiles: the last one of a row or column is about as large as the others
    const int ntx = (g.nbx + side - halo - 1) / (side - halo), nty = (g.nby + side - halo - 1) / (side - halo);
    tc.tx = ((g.nbx + ntx - 1) / ntx + halo + 3) & ~3;
    tc.ty = ((g.nby + nty - 1) / nty + halo + 3) & ~3;
    if (tc.tx < 2 * wp->win || tc.ty < 2 * wp->win || tc.tx * tc.ty < 32) continue;
    const int64_t tw = (int64_t)tc.tx * g.bin, th = (int64_t)tc.ty * g.bin;
    if ((double)tw + sx >= (double)(1 << 24) || (double)th + sy >= (double)(1 << 24)) continue;
    const double cell = std::max(std::ceil(((double)th + sy) / (rows - 2)), (double)(wp->win * g.bin));
    const double units = vtiles * ntx * nty;
    if (units > (double)UINT32_MAX) continue;  // the kernel numbers its units in 32 bits
    const double records = per_px2 * ((double)tw + sx + cell) * ((double)th + sy + cell);
    const double cost = std::ceil(units / di.sms) * (9000.0 + (double)tc.tx * tc.ty * 0.85 * (cb / 8) + records * 2.5);
    if (best != 0 && cost >= best) continue;
    tc.smem = stack_smem_bytes(tc);
    if ((int64_t)tc.smem > budget || !magic_exact(g.bin, std::max(tw, th) - 1)) continue;
    best = cost;
    wp->tc = tc;
    wp->cg.cell = (int32_t)cell;
  }
  if (best == 0) return 0;
  wp->tc.rows = (int)(((double)wp->tc.ty * g.bin + sy) / wp->cg.cell) + 2;
  return wp->tc.rows * (int)E > wp->tc.seg_cap ? 0 : best;
}

// Twice the centre velocity of every group of grp lattice steps, times any dt in
// [0, dT], fits 64 bits.
bool centre_fits(int32_t v0, int32_t dv, uint32_t nv, int grp, int64_t dT) {
  const double most = 2.0 * std::fabs((double)v0) + 2.0 * ((double)nv + grp) * std::fabs((double)dv);
  return most * (double)dT < 9.0e18;
}

}  // namespace

bool plan_windows(const sas_grid_desc& d, uint64_t n, uint32_t n_min, double mean_weight, uint64_t v_begin,
                  uint64_t v_end, const DevInfo& di, const FieldPlan& fp, WindowPlan* wp, int min_bits) {
  const uint32_t E = fp.g.E;
  const uint64_t nv = (uint64_t)d.nvx * d.nvy;
  if (E > (uint32_t)kMaxWindowEpochs || n_min < 2 || n_min > (mean_weight > 0 ? 32768u : 128u)) return false;
  const bool masked = v_begin != 0 || v_end != nv || d.speed_min != 0 || d.speed_max != 0;
  if (masked && nv > ((uint64_t)1 << 24)) return false;
  const double n_v = (double)(v_end - v_begin);
  // GPU cycles of the one-level kernel: 5e-4 per pair with merged reductions (8e-4
  // without), and its counters' finish pass.
  StackArgs sa{};
  fill_stack_args(fp, n_min, n_min, 0, &sa);
  const double counters = n_v * (double)d.nbx * d.nby / ((double)fp.sb * fp.sb);
  const double one_level = (double)n * n_v * (fp.cb == 8 ? (sa.merge ? 5e-4 : 8e-4) : 1.4e-3) +
                           counters * (fp.cb / 32.0) * (6.0 / 32.0 / 2.2 / di.sms);
  // the window search launches five more kernels: about 40000 cycles
  if (one_level < 60000) return false;
  const double hour = (double)fp.dT / (double)fp.g.tph;
  const int64_t unit = d.bin;
  const double density = (double)n / ((double)d.nbx * d.nby * (double)d.bin * d.bin);
  // weighted: 16-bit counters of weights; noise windows by the number of mean weights that reach n_min
  const int cb = mean_weight > 0 ? 16 : min_bits;
  const int n_eq = mean_weight > 0 ? std::max(2, (int)((double)n_min / mean_weight)) : (int)n_min;
  const bool square = std::llabs((int64_t)d.dvx) == std::llabs((int64_t)d.dvy);
  double best = one_level - 40000;
  bool found = false;
  for (int lx = 0; lx <= 3; ++lx)
    for (int ly = 0; ly <= 3; ++ly)
      for (int win = 2; win <= 3; ++win) {
        const int gx = 1 << lx, gy = 1 << ly;
        if (gx * gy == 1 || (square && gx != gy)) continue;
        // steps of a group are 32-bit; twice its centre velocity times dt (k_window_tables) is 64-bit
        if (gx * std::llabs((int64_t)d.dvx) > INT32_MAX || gy * std::llabs((int64_t)d.dvy) > INT32_MAX ||
            !centre_fits(d.vx0, d.dvx, d.nvx, gx, fp.dT) || !centre_fits(d.vy0, d.dvy, d.nvy, gy, fp.dT))
          continue;
        const double hx = 0.5 * (gx - 1) * std::fabs((double)d.dvx) * hour, hy = 0.5 * (gy - 1) * std::fabs((double)d.dvy) * hour;
        const double side = std::ceil(((double)unit + std::max(hx, hy) + 2.0) / (win - 1));
        if (side > (double)(kMaxOwn * unit) || side * win >= (double)(1 << 20)) continue;
        const int64_t P = std::max<int64_t>((int64_t)side, 2), mx = (int64_t)hx + 2, my = (int64_t)hy + 2;
        const int64_t nbx = ((int64_t)d.nbx * d.bin + 2 * mx + P - 1) / P, nby = ((int64_t)d.nby * d.bin + 2 * my + P - 1) / P;
        if (std::llabs((int64_t)d.x_min - mx) >= kLimDomain || std::llabs((int64_t)d.y_min - my) >= kLimDomain ||
            (nbx + 4) * P >= kLimDomain || (nby + 4) * P >= kLimDomain)
          continue;
        // windows that noise alone fills: about 2000 instructions of level 2 each
        const double windows = (n_v / (gx * gy) + 1) * (double)nbx * nby;
        const double lam = density * (double)(win * P) * (double)(win * P);
        const double chance = windows * ((double)n_eq <= lam ? 1.0 : std::exp(std::min(0.0, log_poisson_tail(lam, n_eq))));
        const double level2 = chance * ((mean_weight > 0 ? 3000.0 : 2000.0) / 2.2 / di.sms);
        if (level2 >= best || chance > 4e6) continue;
        WindowPlan w{};
        w.gx = gx;
        w.gy = gy;
        w.win = win;
        w.unit = (int)unit;
        w.g = fp.g;
        w.g.dvx = d.dvx * gx;  // used by the planner only; the shifts come from tables
        w.g.dvy = d.dvy * gy;
        w.g.nvx = (int32_t)div_ceil_u32(d.nvx, (uint32_t)gx);
        w.g.nvy = (int32_t)div_ceil_u32(d.nvy, (uint32_t)gy);
        w.g.smin = w.g.smax = 0;
        w.g.x_min = (int32_t)(d.x_min - mx);
        w.g.y_min = (int32_t)(d.y_min - my);
        w.g.nbx = (int32_t)nbx;
        w.g.nby = (int32_t)nby;
        w.g.bin = (int32_t)P;
        const double level1 = window_tiles(d, n, (v_begin / d.nvx) / gy, ((v_end - 1) / d.nvx) / gy, hour, cb, di, fp, &w);
        if (level1 == 0 || level1 + level2 >= best) continue;
        best = level1 + level2;
        found = true;
        *wp = w;
        wp->list_cap = (uint32_t)std::min<double>(std::max(4.0 * chance, (double)n) + (1 << 18), 1 << 24);
      }
  if (!found) return false;
  wp->masked = masked;
  bucket_grid(d, E, fp.dT, fp.g.tph, &wp->cg);
  while ((uint64_t)E * wp->cg.ncx * wp->cg.ncy > std::max<uint64_t>((uint64_t)1 << 22, 8 * n)) {
    wp->cg.cell *= 2;  // more buckets than the scan over them is worth
    bucket_grid(d, E, fp.dT, fp.g.tph, &wp->cg);
  }
  const double sy = 3.0 * std::fabs((double)wp->g.dvy) * hour + 2.0;
  wp->tc.rows = (int)(((double)wp->tc.ty * wp->g.bin + sy) / wp->cg.cell) + 2;
  wp->nb = (uint64_t)E * wp->cg.ncx * wp->cg.ncy;
  return true;
}

}  // namespace sas
