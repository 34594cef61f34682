// Count stamps of candidates: the input of the candidate vetter.
//
// Stamp of candidate (v_idx, bx, by): 9 x 15 x 15 distinct-epoch counts.  Plane
// q = (dy + 1) * 3 + (dx + 1) is the histogram (Sec. 2.1 step 2) of lattice
// point (kx + dx, ky + dy); element (i, j) is its bin (bx - 7 + j, by - 7 + i).
// Points off the lattice and bins off the domain count 0.
#include <algorithm>

#include "sas_batch.cuh"

namespace sas {

namespace {

constexpr int kStampThreads = 256;
constexpr int kSide = 15;
constexpr int kCells = kSide * kSide;

// Planes of all three lattice rows at once up to 8 words of epochs (65 KB of masks),
// one row at a time beyond (at most 86 KB, at 1024 epochs).
constexpr int kJointWords = 8;
constexpr size_t kStampSmem = (size_t)3 * kCells * (SAS_MAX_EPOCHS / 32) * 4;
static_assert(kStampSmem >= (size_t)9 * kCells * kJointWords * 4, "both forms");
__host__ __device__ inline int rows_per_pass(uint32_t W) { return W <= (uint32_t)kJointWords ? 3 : 1; }
size_t stamp_smem(uint32_t max_e) {  // of any field of up to max_e epochs
  const uint32_t W = (max_e + 31) / 32;
  return std::max((size_t)9 * kCells * std::min<uint32_t>(W, kJointWords), (size_t)3 * kCells * W) * 4;
}
// One candidate's stamp, by one block: in a shared epoch bitmask per plane and cell,
// the epochs of the detections that fall there, then the popcounts.  A thread takes
// an epoch and scans its buckets once for all planes of the pass: the planes' windows
// of 15 x 15 bins differ by the shifts of neighbouring lattice points, a pixel or two.
// (A scan per plane read each bucket nine times; buckets get larger with the number
// of epochs: 4096 stamps after a search of 255 epochs and 1.5 million detections took
// 1352 us, now 604, and of 100 epochs and 300,000 208 us, now 103.)  What bounds it: the
// records read from L2; two or four lanes to an epoch made no difference or cost time.
// Where a lattice step shifts by more than a window, its windows are scanned one by one.
__device__ void stamp_one(const sas_candidate& cd, const SearchGeom& g, const CoarseGeom& cg,
                          const Det* __restrict__ dets, const uint32_t* __restrict__ boff,
                          const uint32_t* __restrict__ ecount, const int32_t* __restrict__ sxt,
                          const int32_t* __restrict__ syt, uint16_t* __restrict__ out, uint32_t* s_mask) {
  const uint32_t W = (g.E + 31) / 32;
  const int R = rows_per_pass(W);
  const int kx = (int)(cd.v_idx % (uint32_t)g.nvx), ky = (int)(cd.v_idx / (uint32_t)g.nvx);
  const int32_t span = kSide * g.bin;
  for (int r0 = 0; r0 < 3; r0 += R) {
    for (uint32_t i = threadIdx.x; i < 3 * R * kCells * W; i += blockDim.x) s_mask[i] = 0;
    __syncthreads();
    for (uint32_t e = threadIdx.x; e < g.E; e += blockDim.x) {
      if (ecount[e] == 0) continue;
      // window origins of the lattice columns and of the pass's rows: bin (bx - 7, by - 7)
      // shifted back to epoch e (points off the lattice: none)
      int32_t ox[3], oy[3];
      uint32_t on_x = 0, on_y = 0;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int kx2 = kx + k - 1, ky2 = ky + r0 + k - 1;
        ox[k] = oy[k] = 0;
        if (kx2 >= 0 && kx2 < g.nvx) {
          ox[k] = g.x_min + ((int32_t)cd.bx - 7) * g.bin + sxt[(size_t)kx2 * g.E + e];
          on_x |= 1u << k;
        }
        if (k < R && ky2 >= 0 && ky2 < g.nvy) {
          oy[k] = g.y_min + ((int32_t)cd.by - 7) * g.bin + syt[(size_t)ky2 * g.E + e];
          on_y |= 1u << k;
        }
      }
      auto bounds = [](const int32_t (&o)[3], uint32_t on, int32_t& lo, int32_t& hi) {
        lo = INT32_MAX;
        hi = INT32_MIN;
#pragma unroll
        for (int k = 0; k < 3; ++k)
          if ((on >> k) & 1u) {
            lo = min(lo, o[k]);
            hi = max(hi, o[k]);
          }
      };
      int32_t lo, hi;
      bounds(ox, on_x, lo, hi);
      const bool apart_x = (int64_t)hi - lo > span;
      bounds(oy, on_y, lo, hi);
      const bool apart_y = (int64_t)hi - lo > span;
      for (uint32_t left_y = on_y; left_y;) {
        const uint32_t ys = apart_y ? left_y & (0u - left_y) : left_y;
        left_y &= ~ys;
        int32_t y0, y1;
        bounds(oy, ys, y0, y1);
        const int cya = max(floor_div32(y0 - cg.gy0, cg.cell), 0);
        const int cyb = min(floor_div32(y1 + span - 1 - cg.gy0, cg.cell), cg.ncy - 1);
        for (uint32_t left_x = on_x; left_x;) {
          const uint32_t xs = apart_x ? left_x & (0u - left_x) : left_x;
          left_x &= ~xs;
          int32_t x0, x1;
          bounds(ox, xs, x0, x1);
          const int cxa = max(floor_div32(x0 - cg.gx0, cg.cell), 0);
          const int cxb = min(floor_div32(x1 + span - 1 - cg.gx0, cg.cell), cg.ncx - 1);
          for (int cy = cya; cy <= cyb && cxa <= cxb; ++cy) {
            const size_t b0 = ((size_t)e * cg.ncy + cy) * cg.ncx;
            const uint32_t k1 = boff[b0 + cxb + 1];
            for (uint32_t k = boff[b0 + cxa]; k < k1; ++k) {
              const Det d = dets[k];
              if ((uint32_t)(d.x - x0) >= (uint32_t)(x1 - x0 + span) || (uint32_t)(d.y - y0) >= (uint32_t)(y1 - y0 + span))
                continue;
#pragma unroll
              for (int r = 0; r < 3; ++r) {
                const uint32_t Y = (uint32_t)(d.y - oy[r]);
                if (!((ys >> r) & 1u) || Y >= (uint32_t)span) continue;
                const int i = (int)(Y / (uint32_t)g.bin), byy = (int)cd.by - 7 + i;
                if (byy < 0 || byy >= g.nby) continue;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                  const uint32_t X = (uint32_t)(d.x - ox[c]);
                  if (!((xs >> c) & 1u) || X >= (uint32_t)span) continue;
                  const int j = (int)(X / (uint32_t)g.bin), bxx = (int)cd.bx - 7 + j;
                  if (bxx < 0 || bxx >= g.nbx) continue;
                  atomicOr(&s_mask[((r * 3 + c) * kCells + i * kSide + j) * W + (e >> 5)], 1u << (e & 31));
                }
              }
            }
          }
        }
      }
    }
    __syncthreads();
    uint16_t* o = out + r0 * 3 * kCells;
    for (int i = threadIdx.x; i < 3 * R * kCells; i += blockDim.x) {
      uint32_t d = 0;
      for (uint32_t w = 0; w < W; ++w) d += __popc(s_mask[i * W + w]);
      o[i] = (uint16_t)min(d, 65535u);
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kStampThreads) k_stamps(
    const sas_candidate* __restrict__ cands, const uint32_t* __restrict__ idx, uint64_t first,
    uint64_t n, SearchGeom g, CoarseGeom cg, const Det* __restrict__ dets,
    const uint32_t* __restrict__ boff, const uint32_t* __restrict__ ecount,
    const int32_t* __restrict__ sxt, const int32_t* __restrict__ syt, uint16_t* __restrict__ out) {
  extern __shared__ uint32_t s_mask[];
  for (uint64_t c = blockIdx.x; c < n; c += gridDim.x) {
    const sas_candidate cd = cands[idx ? (uint64_t)idx[c] : first + c];
    stamp_one(cd, g, cg, dets, boff, ecount, sxt, syt, out + c * 9 * kCells, s_mask);
  }
}

// Stamps of (field[i], cand[i]) items of a batch; the field's own geometry,
// buckets and shift tables.
__global__ void __launch_bounds__(kStampThreads) k_batch_stamps(
    const BatchField* __restrict__ F, const uint32_t* __restrict__ field, const uint32_t* __restrict__ cand,
    uint64_t n, uint16_t* __restrict__ out) {
  extern __shared__ uint32_t s_mask[];
  for (uint64_t c = blockIdx.x; c < n; c += gridDim.x) {
    const BatchField& bf = F[field[c]];
    const sas_candidate cd = bf.cands[cand[c]];
    stamp_one(cd, bf.args.g, bf.args.cg, bf.args.dets, bf.args.boff, bf.ecount, bf.sxt, bf.syt,
              out + c * 9 * kCells, s_mask);
  }
}

}  // namespace

cudaError_t launch_batch_stamps(const BatchField* F, uint32_t max_e, const uint32_t* field, const uint32_t* cand,
                                uint64_t n, uint16_t* out, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const size_t smem = stamp_smem(max_e);
  cudaError_t e = cudaFuncSetAttribute(k_batch_stamps, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStampSmem);
  if (e != cudaSuccess) return e;
  const unsigned blocks = (unsigned)(n < 152ull * 16 ? n : 152ull * 16);
  k_batch_stamps<<<blocks, kStampThreads, smem, s>>>(F, field, cand, n, out);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_stamps(const CandView& v, const uint32_t* idx, uint64_t first, uint64_t count,
                          uint16_t* out, cudaStream_t s) {
  if (count == 0) return cudaSuccess;
  const size_t smem = stamp_smem(v.g.E);
  cudaError_t e = cudaFuncSetAttribute(k_stamps, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStampSmem);
  if (e != cudaSuccess) return e;
  const unsigned blocks = (unsigned)(count < 152ull * 16 ? count : 152ull * 16);
  k_stamps<<<blocks, kStampThreads, smem, s>>>(v.cands, idx, first, count, v.g, v.cg, v.dets, v.boff,
                                                v.ecount, v.sxt, v.syt, out);
  note_launch();
  return cudaGetLastError();
}

}  // namespace sas
