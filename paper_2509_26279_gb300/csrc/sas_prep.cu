// Ingest, bucketing, reference epoch, shift tables and scans (Sec. 2.1 step 1).
#include <algorithm>
#include <climits>

#include "sas_internal.cuh"

namespace sas {

namespace {

constexpr int kPrepThreads = 256;

// a1 + a2 (count phase): validate each detection, count detections per epoch
// (for the reference epoch t0, which is taken over the whole catalog) and per
// spatial bucket.  Detections whose coarse cell lies outside the bucket grid can
// never project into the histogram domain and get no bucket.
__global__ void k_ingest(const int32_t* __restrict__ x, const int32_t* __restrict__ y,
                         const uint16_t* __restrict__ epoch, uint64_t n, uint32_t E,
                         CoarseGeom cg, uint32_t* __restrict__ bucket_count,
                         uint32_t* __restrict__ ecount, uint32_t* __restrict__ bucket_of,
                         uint32_t* __restrict__ flags) {
  extern __shared__ uint32_t s_hist[];  // [E] per-block epoch histogram
  for (uint32_t e = threadIdx.x; e < E; e += blockDim.x) s_hist[e] = 0;
  __syncthreads();
  uint32_t fl = 0;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t e = epoch[i];
    const int32_t xi = x[i], yi = y[i];
    uint32_t b = kInvalidBucket;
    if (e >= E) {
      fl |= kFlagEpoch;
    } else {
      atomicAdd(&s_hist[e], 1u);
      if (xi <= -kLimPos || xi >= kLimPos || yi <= -kLimPos || yi >= kLimPos) {
        fl |= kFlagPos;
      } else {
        const int64_t cx = floor_div64((int64_t)xi - cg.gx0, cg.cell);
        const int64_t cy = floor_div64((int64_t)yi - cg.gy0, cg.cell);
        if (cx >= 0 && cx < cg.ncx && cy >= 0 && cy < cg.ncy) {
          b = (uint32_t)(((uint64_t)e * cg.ncy + (uint64_t)cy) * cg.ncx + (uint64_t)cx);
        } else {
          b = (uint32_t)((uint64_t)E * cg.ncy * cg.ncx);  // overflow bucket: outside the grid
        }
        atomicAdd(&bucket_count[b], 1u);
      }
    }
    bucket_of[i] = b;
  }
  if (fl) atomicOr(flags, fl);
  __syncthreads();
  for (uint32_t e = threadIdx.x; e < E; e += blockDim.x)
    if (s_hist[e]) atomicAdd(&ecount[e], s_hist[e]);
}

// a2 (scatter phase): place each bucketed detection at its bucket's cursor.
__global__ void k_scatter(const int32_t* __restrict__ x, const int32_t* __restrict__ y,
                          const uint16_t* __restrict__ epoch, uint64_t n,
                          const uint32_t* __restrict__ bucket_of, uint32_t* __restrict__ cursor,
                          Det* __restrict__ dets) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t b = bucket_of[i];
    if (b == kInvalidBucket) continue;
    const uint32_t pos = atomicAdd(&cursor[b], 1u);
    Det d;
    d.x = x[i];
    d.y = y[i];
    d.e = epoch[i];
    d.id = (uint32_t)i;
    dets[pos] = d;
  }
}

// Earliest time over the epochs with detections, for a block of whole warps
// (s_min: one entry per warp).
__device__ __forceinline__ long long block_t0(uint32_t E, const int64_t* __restrict__ t,
                                              const uint32_t* __restrict__ ecount, long long* s_min) {
  long long m = LLONG_MAX;
  for (uint32_t e = threadIdx.x; e < E; e += blockDim.x)
    if (ecount[e] > 0 && t[e] < m) m = t[e];
  for (int o = 16; o > 0; o >>= 1) {
    const long long other = __shfl_xor_sync(0xffffffffu, m, o);
    m = other < m ? other : m;
  }
  if ((threadIdx.x & 31) == 0) s_min[threadIdx.x >> 5] = m;
  __syncthreads();
  m = s_min[0];
  for (uint32_t w = 1; w < blockDim.x / 32; ++w) m = s_min[w] < m ? s_min[w] : m;
  return m;
}

// Sec. 2.1 step 1: the reference epoch t0 is the earliest observation time of
// the catalog (over epochs that hold at least one detection); dt[e] = t[e] - t0.
// Sec. 2 Eq. 1-2: the shift of lattice column k at epoch e, s[k][e] =
// floor((v0 + k*dv) * dt[e] / TPH), exact in int64.  One kernel for both axes:
// every block takes the minimum over the (at most 1024) epochs itself, block 0
// also writes dt and t0.
__global__ void __launch_bounds__(kPrepThreads) k_shift_tables(SearchGeom g, const int64_t* __restrict__ t,
                                                               const uint32_t* __restrict__ ecount,
                                                               int64_t* __restrict__ dt, int64_t* __restrict__ t0_out,
                                                               int32_t* __restrict__ sxt, int32_t* __restrict__ syt,
                                                               uint32_t* __restrict__ flags) {
  __shared__ long long s_min[kPrepThreads / 32];
  const long long t0 = block_t0(g.E, t, ecount, s_min);
  if (blockIdx.x == 0) {
    for (uint32_t e = threadIdx.x; e < g.E; e += blockDim.x) dt[e] = ecount[e] > 0 ? (int64_t)(t[e] - t0) : 0;
    if (threadIdx.x == 0) *t0_out = t0;
  }
  const uint64_t nx = (uint64_t)g.nvx * g.E, total = nx + (uint64_t)g.nvy * g.E;
  uint32_t fl = 0;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < total; i += (uint64_t)gridDim.x * blockDim.x) {
    const bool y = i >= nx;
    const uint64_t at = y ? i - nx : i;
    const uint32_t k = (uint32_t)(at / g.E), e = (uint32_t)(at % g.E);
    const int64_t v = y ? (int64_t)g.vy0 + (int64_t)k * g.dvy : (int64_t)g.vx0 + (int64_t)k * g.dvx;
    const bool used = ecount[e] > 0;
    const int64_t s = used ? floor_div64(v * (t[e] - t0), g.tph) : 0;
    int32_t sv = 0;
    if (s <= -kLimDomain || s >= kLimDomain) fl |= kFlagShift; else sv = (int32_t)s;
    (y ? syt : sxt)[at] = sv;
  }
  if (fl) atomicOr(flags, fl);
}

// ---- exclusive scan: block sums, then apply; beyond kScanSelf tiles the sums are
// scanned first, below it every apply block adds up the sums before its own (one
// launch less) -----------------------------------------------------------------
constexpr uint64_t kScanSelf = 2048;

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

template <typename T>
__device__ T block_exclusive_scan(T v, T* s_warp, T* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  T inc = v;
  for (int o = 1; o < 32; o <<= 1) {
    T n = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += n;
  }
  if (lane == 31) s_warp[w] = inc;
  __syncthreads();
  if (w == 0) {
    const int nw = blockDim.x >> 5;
    T s = lane < nw ? s_warp[lane] : T(0);
    T si = s;
    for (int o = 1; o < 32; o <<= 1) {
      T n = __shfl_up_sync(0xffffffffu, si, o);
      if (lane >= o) si += n;
    }
    if (lane < nw) s_warp[lane] = si - s;
    if (lane == nw - 1) s_warp[32] = si;
  }
  __syncthreads();
  const T r = s_warp[w] + inc - v;
  if (total) *total = s_warp[32];
  __syncthreads();
  return r;
}

template <typename Tin, typename Tout>
__global__ void k_scan_reduce(const Tin* __restrict__ in, uint64_t n, Tout* __restrict__ sums) {
  __shared__ Tout s_warp[33];
  const uint64_t base = (uint64_t)blockIdx.x * kScanTile;
  Tout acc = 0;
  for (int k = 0; k < kScanItems; ++k) {
    const uint64_t i = base + (uint64_t)threadIdx.x * kScanItems + k;
    if (i < n) acc += (Tout)in[i];
  }
  Tout total;
  block_exclusive_scan<Tout>(acc, s_warp, &total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// One block scans the block sums in place (any count, carried across rounds).
template <typename Tout>
__global__ void k_scan_top(Tout* __restrict__ sums, uint64_t nb) {
  __shared__ Tout s_warp[33];
  Tout carry = 0;
  for (uint64_t base = 0; base < nb; base += blockDim.x) {
    const uint64_t i = base + threadIdx.x;
    const Tout v = i < nb ? sums[i] : Tout(0);
    Tout total;
    const Tout ex = block_exclusive_scan<Tout>(v, s_warp, &total);
    if (i < nb) sums[i] = carry + ex;
    carry += total;
  }
}

// Sum of the block sums before this block's (self), or its scanned sum.
template <typename Tout>
__device__ Tout tiles_before(const Tout* __restrict__ sums, bool self, Tout* s_warp) {
  if (!self) return sums[blockIdx.x];
  Tout v = 0, total;
  for (uint32_t i = threadIdx.x; i < blockIdx.x; i += blockDim.x) v += sums[i];
  block_exclusive_scan<Tout>(v, s_warp, &total);
  return total;
}

template <typename Tin, typename Tout>
__global__ void k_scan_apply(const Tin* __restrict__ in, uint64_t n, const Tout* __restrict__ sums, bool self,
                             Tout* __restrict__ out, Tout* __restrict__ out2) {
  __shared__ Tout s_warp[33];
  const uint64_t base = (uint64_t)blockIdx.x * kScanTile;
  Tout v[kScanItems];
  Tout acc = 0;
  for (int k = 0; k < kScanItems; ++k) {
    const uint64_t i = base + (uint64_t)threadIdx.x * kScanItems + k;
    v[k] = i < n ? (Tout)in[i] : Tout(0);
    acc += v[k];
  }
  const Tout before = tiles_before<Tout>(sums, self, s_warp);
  Tout total;
  Tout run = block_exclusive_scan<Tout>(acc, s_warp, &total) + before;
  for (int k = 0; k < kScanItems; ++k) {
    const uint64_t i = base + (uint64_t)threadIdx.x * kScanItems + k;
    if (i < n) {
      out[i] = run;
      if (out2) out2[i] = run;
    }
    run += v[k];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == blockDim.x - 1) out[n] = run;
}

template <typename Tin, typename Tout>
cudaError_t scan_impl(const Tin* in, Tout* out, Tout* out2, uint64_t n, Tout* scratch, cudaStream_t s) {
  if (n == 0) return cudaMemsetAsync(out, 0, sizeof(Tout), s);
  const uint64_t nb = (n + kScanTile - 1) / kScanTile;
  const bool self = nb <= kScanSelf;
  if (nb > 1) {
    k_scan_reduce<Tin, Tout><<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, scratch);
    note_launch();
  }
  if (!self) {
    k_scan_top<Tout><<<1, kScanThreads, 0, s>>>(scratch, nb);
    note_launch();
  }
  k_scan_apply<Tin, Tout><<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, scratch, self, out, out2);
  note_launch();
  return cudaGetLastError();
}

// ---- id offsets and candidate records of sorted keys ------------------------------

// The raw count of key i is the low half of ~a.
__global__ void k_raw_sums(const Key* __restrict__ keys, uint32_t n, unsigned long long* __restrict__ sums) {
  __shared__ unsigned long long s_warp[33];
  const uint32_t i = blockIdx.x * kScanThreads + threadIdx.x;
  unsigned long long total;
  block_exclusive_scan<unsigned long long>(i < n ? (unsigned long long)(~(uint32_t)keys[i].a) : 0ull, s_warp, &total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void k_candidates(const Key* __restrict__ keys, uint32_t n, const unsigned long long* __restrict__ sums,
                             bool self, unsigned long long* __restrict__ id_off, sas_candidate* __restrict__ out,
                             unsigned long long* __restrict__ n_ids) {
  __shared__ unsigned long long s_warp[33];
  const uint32_t i = blockIdx.x * kScanThreads + threadIdx.x;
  Key k{};
  uint32_t raw = 0;
  if (i < n) {
    k = keys[i];
    raw = ~(uint32_t)k.a;
  }
  const unsigned long long before = tiles_before<unsigned long long>(sums, self, s_warp);
  const unsigned long long off = block_exclusive_scan<unsigned long long>(raw, s_warp, nullptr) + before;
  if (i >= n) return;
  sas_candidate c;
  c.v_idx = (uint32_t)(k.b >> 32);
  c.by = (uint32_t)k.b;
  c.bx = k.c;
  c.count = ~(uint32_t)(k.a >> 32);
  c.raw = c.id_len = raw;
  c.id_off = off;
  out[i] = c;
  id_off[i] = off;
  if (i == n - 1) *n_ids = off + raw;
}

// Largest weight and sum of weights, one atomic pair per block.
__global__ void k_weight_stats(const uint8_t* __restrict__ w, uint64_t n, unsigned long long* __restrict__ out) {
  uint32_t top = 0;
  unsigned long long sum = 0;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    top = max(top, (uint32_t)w[i]);
    sum += w[i];
  }
  __shared__ unsigned long long s_sum[kPrepThreads / 32];
  __shared__ uint32_t s_top[kPrepThreads / 32];
  top = __reduce_max_sync(0xffffffffu, top);
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if ((threadIdx.x & 31) == 0) {
    s_top[threadIdx.x >> 5] = top;
    s_sum[threadIdx.x >> 5] = sum;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < kPrepThreads / 32; ++i) {
      top = max(top, s_top[i]);
      sum += s_sum[i];
    }
    atomicMax(&out[0], (unsigned long long)top);
    atomicAdd(&out[1], sum);
  }
}

unsigned grid_for(uint64_t n, int threads) {
  uint64_t b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > 152ull * 64) b = 152ull * 64;
  return (unsigned)b;
}

}  // namespace

size_t scan_scratch_elems(uint64_t n) { return (size_t)((n + kScanTile - 1) / kScanTile) + 1; }

cudaError_t launch_scan_u32(const uint32_t* in, uint32_t* out, uint64_t n, uint32_t* scratch, cudaStream_t s,
                            uint32_t* out2) {
  return scan_impl<uint32_t, uint32_t>(in, out, out2, n, scratch, s);
}

cudaError_t launch_candidates(const Key* keys, uint32_t n, unsigned long long* id_off, unsigned long long* scratch,
                              sas_candidate* out, unsigned long long* n_ids, cudaStream_t s) {
  if (n == 0) return cudaSuccess;  // *n_ids stays zero
  const uint32_t nb = (n + kScanThreads - 1) / kScanThreads;
  const bool self = nb <= kScanSelf;
  if (nb > 1) {
    k_raw_sums<<<nb, kScanThreads, 0, s>>>(keys, n, scratch);
    note_launch();
  }
  if (!self) {
    k_scan_top<unsigned long long><<<1, kScanThreads, 0, s>>>(scratch, nb);
    note_launch();
  }
  k_candidates<<<nb, kScanThreads, 0, s>>>(keys, n, scratch, self, id_off, out, n_ids);
  note_launch();
  return cudaGetLastError();
}
size_t candidates_scratch_elems(uint64_t n) { return (size_t)((n + kScanThreads - 1) / kScanThreads) + 1; }

cudaError_t launch_ingest(const int32_t* x, const int32_t* y, const uint16_t* epoch, uint64_t n,
                          uint32_t E, CoarseGeom cg, uint32_t* bucket_count, uint32_t* ecount,
                          uint32_t* bucket_of, uint32_t* flags, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  k_ingest<<<grid_for(n, kPrepThreads), kPrepThreads, E * sizeof(uint32_t), s>>>(
      x, y, epoch, n, E, cg, bucket_count, ecount, bucket_of, flags);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_scatter(const int32_t* x, const int32_t* y, const uint16_t* epoch, uint64_t n,
                           const uint32_t* bucket_of, uint32_t* cursor, Det* dets,
                           cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  k_scatter<<<grid_for(n, kPrepThreads), kPrepThreads, 0, s>>>(x, y, epoch, n, bucket_of, cursor,
                                                                dets);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_weight_stats(const uint8_t* w, uint64_t n, unsigned long long* out, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, 16, s);
  if (e != cudaSuccess) return e;
  k_weight_stats<<<(unsigned)std::min<uint64_t>((n + 8 * kPrepThreads - 1) / (8 * kPrepThreads), 304), kPrepThreads, 0, s>>>(w, n, out);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_shift_tables(const SearchGeom& g, const int64_t* t, const uint32_t* ecount, int64_t* dt, int64_t* t0,
                                int32_t* sxt, int32_t* syt, uint32_t* flags, cudaStream_t s) {
  k_shift_tables<<<grid_for(((uint64_t)g.nvx + g.nvy) * g.E, kPrepThreads), kPrepThreads, 0, s>>>(
      g, t, ecount, dt, t0, sxt, syt, flags);
  note_launch();
  return cudaGetLastError();
}

}  // namespace sas
