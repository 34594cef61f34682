// Candidate vetter: a small CNN that scores a candidate from its count stamp,
// trained and run on the GPU (BF16 weights and activations, FP32 accumulation).
//
// Filtering the search results better is the paper's own suggestion for going
// fainter (Sec. 5); this network is that filter.  Network (input = count / 16):
//   conv1 9->32 3x3 valid + ReLU (15 -> 13), conv2 32->32 (13 -> 11) + ReLU,
//   conv3 32->32 (11 -> 9) + ReLU, flatten (channel, row, column),
//   fc1 2592 -> 64 + ReLU, fc2 64 -> 1 = logit;  loss: mean BCE with logits.
// Flat parameter order: conv1.w [32,9,3,3], conv1.b, conv2.w [32,32,3,3],
// conv2.b, conv3.w, conv3.b, fc1.w [64,2592], fc1.b, fc2.w [64], fc2.b.
//
// Numerics: weights are used as BF16 copies of FP32 master values; every stored
// activation (input, conv outputs, fc1 output) is rounded to BF16; products are
// exact in FP32 and accumulate in FP32.  Back-propagated deltas and weight
// gradients are FP32.  Weight gradients are summed per block over a fixed
// stamp-to-block assignment and then over blocks in a fixed order, so a
// gradient is bit-reproducible for a given batch.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "sas_internal.cuh"
#include "sas_tc.cuh"

struct sas_vet {
  int device;
  int sms;               // the device's SMs
  uint32_t max_batch;
  uint64_t step;
  float beta1, beta2, eps;
  // parameters
  float* master;
  float* m;
  float* v;
  float* grad;
  __nv_bfloat16* wb;     // BF16 copy in the flat order
  // activations and deltas of one batch
  __nv_bfloat16* a1;     // [B][32][13][13]
  __nv_bfloat16* a2;     // [B][32][11][11]
  __nv_bfloat16* a3;     // [B][2592]
  __nv_bfloat16* a4;     // [B][64]
  float* logits;         // [B]
  float* fcpart;         // [kFcSplit][64][B rounded up to 128] fc1 partial sums
  float* g4;             // [B][64]
  float* g3;             // [B][2592]
  float* g2;             // [B][32][11][11]
  float* g1;             // [B][32][13][13]
  float* partial;        // per-block weight-gradient partial sums, one part per conv layer
  float* lpart;          // per-block sums of the loss and the fc2 gradients
  float* loss;           // [1]
  uint32_t* status;      // [1] nonzero: a tensor-core wait gave up (sas_vet_check)
};

namespace sas {
namespace vet {

constexpr int kS = 15, kQ = 9, kCh = 32;
constexpr int kH1 = 13, kH2 = 11, kH3 = 9;
constexpr int kF = kCh * kH3 * kH3;  // 2592
constexpr int kHid = 64;
constexpr int kW1 = 0, kB1 = kW1 + kCh * kQ * 9, kW2 = kB1 + kCh, kB2 = kW2 + kCh * kCh * 9;
constexpr int kW3 = kB2 + kCh, kB3 = kW3 + kCh * kCh * 9, kWf1 = kB3 + kCh, kBf1 = kWf1 + kHid * kF;
constexpr int kWf2 = kBf1 + kHid, kBf2 = kWf2 + kHid, kNParams = kBf2 + 1;
static_assert(kNParams == 187137, "parameter layout");

constexpr int kBackBlocks = 304;      // blocks (and partial sums) of the conv backward kernels: two per SM
constexpr int kPartialStride = kCh * kCh * 9 + kCh;  // >= parts * weights + biases of any layer
constexpr uint32_t kFc1Slices = 14;                  // stamp slices of the fc1 weight gradient
static_assert((size_t)kFc1Slices * (kHid * kF + kHid) <= (size_t)kBackBlocks * kPartialStride,
              "fc1 slices fit the partial buffer");

__device__ __forceinline__ float ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
// Two values rounded to BF16 in one word (one instruction).
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// ---- forward on the tensor cores: the three convolutions as implicit GEMMs ---
//
// Per stamp and layer: D[pixel][out] = sum over taps (dy, dx) and input channels
// c of A[pixel + dy * W + dx][c] * w[out][c][dy][dx], with A the layer's input
// (W x W pixels, row r = y * W + x) and D computed over the padded output grid
// (rows y * W + x for x < W; the columns x >= W - 2 are not outputs and are
// dropped).  A sits in shared memory as [8-channel chunk][row][8 channels], so
// its rows are 16 bytes apart and the operand of tap (dy, dx) is the same
// buffer started dy * W + dx rows later: no im2col is built.  Each tap of each
// 128-row tile is one tcgen05.mma per 16 input channels (BF16 x BF16 -> FP32 in
// TMEM), all issued by one thread; every warp then reads its TMEM lanes back for
// bias + ReLU + BF16 rounding straight into the next layer's input layout.
// Products are exact in FP32 and the sums accumulate in FP32.

//
// Four stamps are in flight per SM: one CTA of four groups of 8 warps, each with its
// own buffers, TMEM columns, mbarrier and named barrier, around one copy of the
// weights (46 of 198 KB).  A group's chain -- build, MMAs, wait, TMEM loads, store, three
// times a stamp -- is latency, which the other groups' work hides; with two CTAs of
// 16 warps and a copy of the weights each, two stamps were in flight, the tensor
// pipe 24 % and the issue slots 35 % busy.
constexpr int kTcGroups = 4, kTcGrp = 256;  // 8 warps: 4 TMEM lane quadrants x 2 sixteen-channel halves
constexpr int kTcThreads = kTcGroups * kTcGrp;
constexpr int kTcRows0 = 288;     // x0: 15 x 15 pixels; tiles read up to row 2 * 128 - 1 + 2 * 15 + 2
constexpr int kTcRows1 = 288;     // a1: 13 x 13 pixels; up to row 2 * 128 - 1 + 2 * 13 + 2
constexpr int kTcRows2 = 160;     // a2: 11 x 11 pixels; up to row 127 + 2 * 11 + 2
constexpr int kTcW1 = 9 * kCh * 16 * 2;   // per tap: 32 outputs x 16 input channels (9 real)
constexpr int kTcW23 = 9 * kCh * kCh * 2; // per tap: 32 x 32
constexpr int kSmW1 = 0;
constexpr int kSmW2 = kSmW1 + kTcW1;
constexpr int kSmW3 = kSmW2 + kTcW23;
constexpr int kSmBias = kSmW3 + kTcW23;
constexpr int kSmBar = kSmBias + 3 * kCh * 4;             // one mbarrier per group, then the TMEM base
constexpr int kSmGrp = (kSmBar + 8 * kTcGroups + 16 + 127) / 128 * 128;
constexpr int kGrX0 = 0;                                   // within a group's buffers
constexpr int kGrA1 = kGrX0 + 2 * kTcRows0 * 16;
constexpr int kGrA2 = kGrA1 + 4 * kTcRows1 * 16;
constexpr int kGrBytes = kGrA2 + 4 * kTcRows2 * 16;
constexpr int kTcSmem = kSmGrp + kTcGroups * kGrBytes;
constexpr int kTcTmemCols = 512, kTcGrpCols = 128;  // per group: conv1 tiles at columns 0, 32; conv2 at 64, 96; conv3 at 0
static_assert(kTcRows0 >= 2 * 128 + 2 * kS + 2 && kTcRows1 >= 2 * 128 + 2 * kH1 + 2 &&
                  kTcRows2 >= 128 + 2 * kH2 + 2, "shifted windows stay inside the buffers");
static_assert(kSmW1 % 128 == 0 && kSmW2 % 128 == 0 && kSmW3 % 128 == 0 && kGrA1 % 16 == 0 &&
                  kGrA2 % 16 == 0 && kGrBytes % 128 == 0, "operand alignment");
static_assert(kTcSmem <= 226 * 1024, "one CTA per SM");

// Barrier of one group of kTcGrp threads; returns whether any of them passed `bad`.
__device__ __forceinline__ bool group_sync_or(int group, bool bad) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\tbar.red.or.pred p, %2, %3, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)bad), "r"(group + 1), "n"(kTcGrp)
      : "memory");
  return r != 0;
}
__device__ __forceinline__ void group_sync(int group) {
  asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(kTcGrp) : "memory");
}

// Per-tap weights of a layer as the B operand: B_t[o][c] = w[o][c][t]; kc 16-byte
// chunks per row (K = 8 kc; columns c >= cin stay as they are).  Read in memory order.
__device__ void tc_load_w_taps(const __nv_bfloat16* __restrict__ w, int cin, int kc, unsigned char* dst) {
  const int per_tap = kCh * kc * 8;
  for (int i = threadIdx.x; i < kCh * cin * 9; i += blockDim.x) {
    const int o = i / (cin * 9), j = i - o * (cin * 9), c = j / 9, t = j - c * 9;
    *reinterpret_cast<__nv_bfloat16*>(dst + t * per_tap * 2 + tc::cm_offset(o, c, kc)) = w[i];
  }
}

// The MMAs of one layer (thread 0): NT tiles of 128 output rows, 9 taps, KS
// steps of 16 input channels; input rows R per chunk, input width W.
template <int NT, int KS, int R, int W>
__device__ __forceinline__ void tc_conv_mma(uint32_t a_base, uint32_t w_base, uint32_t tmem_col) {
  constexpr uint32_t idesc = tc::idesc_bf16(128, 32);
  constexpr uint32_t per_tap = kCh * KS * 2 * 16;  // bytes of one tap's B operand
#pragma unroll
  for (int t = 0; t < NT; ++t)
    for (int tap = 0; tap < 9; ++tap) {
      const uint32_t shift = (uint32_t)((tap / 3) * W + (tap % 3));
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        const uint64_t ad = tc::smem_desc_strided(a_base + (uint32_t)(2 * ks * R * 16) + (t * 128u + shift) * 16u,
                                                  (uint32_t)(R * 16), 128u);
        const uint64_t bd = tc::smem_desc(w_base + (uint32_t)tap * per_tap + (uint32_t)(2 * ks * 128), 2 * KS);
        tc::mma_bf16(tmem_col + (uint32_t)(t * 32), ad, bd, idesc, (tap | ks) != 0);
      }
    }
}

// Bias, ReLU and BF16 rounding of a layer's D (NT tiles at TMEM column tmem_col)
// over the padded grid of width W (outputs: W - 2 x W - 2) into the next layer's
// input layout (rows (W - 2) * y + x, Rn rows per chunk) and, optionally, the
// global activation [ch][W-2][W-2].
template <int NT, int W, int Rn>
__device__ __forceinline__ void tc_conv_epi(uint32_t tmem_col, const float* bias, unsigned char* next,
                                            __nv_bfloat16* out_g) {
  constexpr int HO = W - 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = warp & 3, h = (warp >> 2) & 1;
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    float v[16];
    tc::ld16(tmem_col + ((uint32_t)(q * 32) << 16) + (uint32_t)(t * 32 + h * 16), v);
    const int m = t * 128 + q * 32 + lane, y = m / W, x = m - y * W;
    if (y < HO && x < HO) {
      const int p = y * HO + x;
      uint32_t pk[8];
#pragma unroll
      for (int j = 0; j < 16; j += 2) {
        pk[j / 2] = pack_bf16(fmaxf(v[j] + bias[h * 16 + j], 0.f), fmaxf(v[j + 1] + bias[h * 16 + j + 1], 0.f));
        if (out_g) {
          uint16_t* g = reinterpret_cast<uint16_t*>(out_g) + (h * 16 + j) * HO * HO + p;
          g[0] = (uint16_t)pk[j / 2];
          g[HO * HO] = (uint16_t)(pk[j / 2] >> 16);
        }
      }
      if (next) {
        *reinterpret_cast<uint4*>(next + (2 * h * Rn + p) * 16) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
        *reinterpret_cast<uint4*>(next + ((2 * h + 1) * Rn + p) * 16) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
      }
    }
  }
}

// One layer of a group: operand visible to the tensor core, MMAs by its first
// thread, bounded wait, epilogue.  Returns false (group-uniform) when the wait gave up.
template <int NT, int KS, int R, int W, int Rn>
__device__ __forceinline__ bool tc_conv_layer(int group, const unsigned char* in, const unsigned char* w,
                                              uint32_t tmem_col, uint64_t* bar, uint32_t& phase, const float* bias,
                                              unsigned char* next, __nv_bfloat16* out_g) {
  tc::fence_smem_to_async();
  tc::fence_before_sync();
  group_sync(group);
  if ((threadIdx.x & (kTcGrp - 1)) == 0) {
    tc::fence_after_sync();
    tc_conv_mma<NT, KS, R, W>(tc::smem_u32(in), tc::smem_u32(w), tmem_col);
    tc::commit(bar);
  }
  const bool ok = tc::mbar_wait(bar, phase, 1u << 22);
  phase ^= 1u;
  if (group_sync_or(group, !ok)) return false;
  tc::fence_after_sync();
  tc_conv_epi<NT, W, Rn>(tmem_col, bias, next, out_g);
  tc::fence_before_sync();
  return true;
}

__global__ void __launch_bounds__(kTcThreads, 1) k_conv_fwd_tc(const uint16_t* __restrict__ stamps,
                                                               const uint32_t* __restrict__ idx, uint32_t n,
                                                               const __nv_bfloat16* __restrict__ wb,
                                                               __nv_bfloat16* a1g, __nv_bfloat16* a2g,
                                                               __nv_bfloat16* __restrict__ a3g,
                                                               uint32_t* __restrict__ status) {
  extern __shared__ __align__(1024) unsigned char smc[];
  float* bias = reinterpret_cast<float*>(smc + kSmBias);
  const int tid = threadIdx.x, group = tid / kTcGrp, gt = tid & (kTcGrp - 1);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smc + kSmBar) + group;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smc + kSmBar + 8 * kTcGroups);
  unsigned char* buf = smc + kSmGrp + group * kGrBytes;
  if (tid < 32) tc::tmem_alloc(tslot, kTcTmemCols);
  if (gt == 0) tc::mbar_init(bar, 1);
  // conv1's weights and the activation buffers: what is never written (channel and
  // row padding) stays zero
  for (int i = tid; i < kSmW2 / 16; i += kTcThreads) reinterpret_cast<uint4*>(smc)[i] = make_uint4(0, 0, 0, 0);
  for (int i = tid; i < kTcGroups * kGrBytes / 16; i += kTcThreads)
    reinterpret_cast<uint4*>(smc + kSmGrp)[i] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  tc_load_w_taps(wb + kW1, kQ, 2, smc + kSmW1);
  tc_load_w_taps(wb + kW2, kCh, 4, smc + kSmW2);
  tc_load_w_taps(wb + kW3, kCh, 4, smc + kSmW3);
  if (tid < 3 * kCh) {
    const int l = tid / kCh, o = tid % kCh;
    bias[tid] = ld(wb + (l == 0 ? kB1 : l == 1 ? kB2 : kB3) + o);
  }
  tc::fence_smem_to_async();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tslot + (uint32_t)(group * kTcGrpCols);
  uint32_t phase = 0;
  // A thread builds rows (8-channel chunk, pixel) gt and gt + 256 of x0, 16 bytes each,
  // and holds the next stamp's counts while the current one runs.
  constexpr int kPix = kS * kS;
  uint32_t nxt[2][4];
  auto fetch = [&](uint32_t b) {
    if (b >= n) return;
    const uint16_t* st = stamps + (size_t)(idx ? idx[b] : b) * kQ * kPix;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int it = gt + r * kTcGrp, chunk = it / kPix, p = it - chunk * kPix;
#pragma unroll
      for (int c = 0; c < 8; c += 2) {
        const uint32_t v0 = chunk == 0 || (chunk == 1 && c == 0) ? st[(chunk * 8 + c) * kPix + p] : 0u;
        const uint32_t v1 = chunk == 0 ? st[(c + 1) * kPix + p] : 0u;
        nxt[r][c / 2] = v0 | (v1 << 16);
      }
    }
  };
  const uint32_t first = blockIdx.x + (uint32_t)group * gridDim.x, stride = kTcGroups * gridDim.x;
  fetch(first);
  for (uint32_t b = first; b < n; b += stride) {
    // x0[chunk][row][channel] = count / 16 in BF16 (exact for counts <= 256 * 16)
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int it = gt + r * kTcGrp, chunk = it / kPix, p = it - chunk * kPix;
      if (chunk < 2) {
        uint32_t pk[4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
          // (2^23 + count) / 16 - 2^19 = count / 16, exactly: no integer conversion
          pk[c] = pack_bf16(fmaf(__uint_as_float(0x4b000000u | (nxt[r][c] & 0xffffu)), 0.0625f, -524288.f),
                            fmaf(__uint_as_float(0x4b000000u | (nxt[r][c] >> 16)), 0.0625f, -524288.f));
        reinterpret_cast<uint4*>(buf + kGrX0)[chunk * kTcRows0 + p] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
      }
    }
    fetch(b + stride);
    if (!tc_conv_layer<2, 1, kTcRows0, kS, kTcRows1>(group, buf + kGrX0, smc + kSmW1, tmem, bar, phase, bias, buf + kGrA1,
                                                     a1g ? a1g + (size_t)b * kCh * kH1 * kH1 : nullptr) ||
        !tc_conv_layer<2, 2, kTcRows1, kH1, kTcRows2>(group, buf + kGrA1, smc + kSmW2, tmem + 64, bar, phase, bias + kCh,
                                                      buf + kGrA2, a2g ? a2g + (size_t)b * kCh * kH2 * kH2 : nullptr) ||
        !tc_conv_layer<1, 2, kTcRows2, kH2, 1>(group, buf + kGrA2, smc + kSmW3, tmem, bar, phase, bias + 2 * kCh, nullptr,
                                               a3g + (size_t)b * kF)) {
      if (gt == 0) atomicOr(status, 1u);
      break;
    }
    // (the next stamp's x0 was read by MMAs that two waits have seen complete, and its
    // first MMAs follow a group barrier behind this epilogue's TMEM loads)
  }
  tc::fence_before_sync();
  __syncthreads();
  if (tid < 32) tc::tmem_free(*tslot, kTcTmemCols);
}

// ---- forward: fc1 on the tensor cores, fc2 in the epilogue --------------------
//
// D[stamp][j] = sum_k a3[stamp][k] * fc1.w[j][k]: M = 128 stamps per block,
// N = 64, K = 2592 in 27 blocks of 96, split over kFcSplit blocks along K so
// that a batch of 4096 stamps keeps 128 SMs busy.  Both operands are
// K-contiguous in global memory; 16-byte rows of core matrices go to the no-swizzle
// K-major layout of one of three stages by asynchronous copies, two blocks ahead of
// the MMAs (one mbarrier per stage, bounded waits); what bounds a block is the
// latency of its 7 K blocks, which copies through registers took one after another
// (41 us for 512 as for 4096 stamps).  Each block
// writes its FP32 partial D column-major; k_fc_epi adds the kFcSplit partials
// in a fixed order, adds the bias, applies ReLU, rounds to BF16, stores a4 and
// forms the logit with fc2 in a fixed order.
constexpr int kFcTcRows = 128, kFcTcKB = 96, kFcTcKC = kFcTcKB / 8, kFcTcNB = kF / kFcTcKB;
constexpr int kFcTcThreads = 256, kFcTcStages = 3, kFcSplit = 4;
constexpr int kFcTcA = kFcTcRows * kFcTcKB * 2, kFcTcB = kHid * kFcTcKB * 2;
constexpr int kFcTcStage = kFcTcA + kFcTcB;
constexpr int kFcTcSmem = kFcTcStages * kFcTcStage + 8 * kFcTcStages + 16;
static_assert(kF % kFcTcKB == 0, "fc1 K blocks");

// part[s][j][stamp] (stamps padded to whole 128-row tiles: ld = tiles * 128)
__global__ void __launch_bounds__(kFcTcThreads) k_fc_fwd_tc(const __nv_bfloat16* __restrict__ a3g, uint32_t n,
                                                            const __nv_bfloat16* __restrict__ wb,
                                                            float* __restrict__ part, uint32_t ldp,
                                                            uint32_t* __restrict__ status) {
  extern __shared__ __align__(1024) unsigned char smf[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(smf + kFcTcStages * kFcTcStage);  // [kFcTcStages]
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + kFcTcStages);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t b0 = blockIdx.x * kFcTcRows;
  const int sp = blockIdx.y;
  const int kb_lo = sp * kFcTcNB / kFcSplit, kb_hi = (sp + 1) * kFcTcNB / kFcSplit;
  if (tid < 32) tc::tmem_alloc(tslot, kHid);
  if (tid == 0)
    for (int st = 0; st < kFcTcStages; ++st) tc::mbar_init(bar + st, 1);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tslot;
  const uint4* a3v = reinterpret_cast<const uint4*>(a3g);
  const uint4* w1v = reinterpret_cast<const uint4*>(wb + kWf1);
  constexpr uint32_t idesc = tc::idesc_bf16(kFcTcRows, kHid);
  const int nkb = kb_hi - kb_lo;
  auto load = [&](int l) {  // K block l of this block's into its stage; one copy group
    if (l < nkb) {
      unsigned char* A = smf + (l % kFcTcStages) * kFcTcStage;
      unsigned char* B = A + kFcTcA;
      const int k8 = (kb_lo + l) * kFcTcKC;  // first 16-byte chunk of the block along K
      for (int i = tid; i < kFcTcRows * kFcTcKC; i += kFcTcThreads) {
        const int r = i / kFcTcKC, c = i - r * kFcTcKC;
        const bool in = b0 + r < n;
        tc::cp16(A + tc::cm_offset(r, c * 8, kFcTcKC), a3v + (in ? (size_t)(b0 + r) * (kF / 8) + k8 + c : 0), in);
      }
      for (int i = tid; i < kHid * kFcTcKC; i += kFcTcThreads) {
        const int r = i / kFcTcKC, c = i - r * kFcTcKC;
        tc::cp16(B + tc::cm_offset(r, c * 8, kFcTcKC), w1v + (size_t)r * (kF / 8) + k8 + c, true);
      }
    }
    tc::cp_commit();
  };
  uint32_t ph[kFcTcStages] = {};
  bool ok = true;
  load(0);
  load(1);
  for (int l = 0; l < nkb && ok; ++l) {
    const int st = l % kFcTcStages, nx = (l + 2) % kFcTcStages;
    if (l + 2 >= kFcTcStages && l + 2 < nkb) {  // the MMAs that read stage nx are done
      ok = tc::mbar_wait(bar + nx, ph[nx], 1u << 22);
      ph[nx] ^= 1u;
      if (__syncthreads_or(!ok)) {
        ok = false;
        break;
      }
    }
    load(l + 2);
    tc::cp_wait<2>();  // block l has arrived
    tc::fence_smem_to_async();
    tc::fence_before_sync();
    __syncthreads();
    if (tid == 0) {
      tc::fence_after_sync();
      const uint32_t a0 = tc::smem_u32(smf + st * kFcTcStage), w0 = a0 + kFcTcA;
#pragma unroll
      for (int ks = 0; ks < kFcTcKC / 2; ++ks)
        tc::mma_bf16(tmem, tc::smem_desc(a0 + (uint32_t)(2 * ks * 128), kFcTcKC),
                     tc::smem_desc(w0 + (uint32_t)(2 * ks * 128), kFcTcKC), idesc, (l > 0 || ks > 0) ? 1u : 0u);
      tc::commit(bar + st);
    }
  }
  tc::cp_wait<0>();
  if (ok) {  // one commit outstanding on every stage that was used
    const int used = min(nkb, kFcTcStages);
    for (int st = 0; st < used && ok; ++st) {
      ok = tc::mbar_wait(bar + st, ph[st], 1u << 22);
      ph[st] ^= 1u;
    }
    ok = !__syncthreads_or(!ok);
  }
  if (!ok) {
    if (tid == 0) atomicOr(status, 1u);
  } else {
    tc::fence_after_sync();
    const int q = warp & 3, h = warp >> 2;  // lane quadrant, column half
    const uint32_t b = b0 + (uint32_t)(q * 32 + lane);
    float* out = part + (size_t)sp * kHid * ldp;
#pragma unroll
    for (int c = h * 32; c < h * 32 + 32; c += 16) {
      float v[16];
      tc::ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c, v);
#pragma unroll
      for (int jj = 0; jj < 16; ++jj) out[(size_t)(c + jj) * ldp + b] = v[jj];
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (tid < 32) tc::tmem_free(tmem, kHid);
}

// 32 stamps x 8 groups of 8 hidden units per block: the partial sums in split
// order, bias, ReLU, BF16, then fc2 -- each group's products in order, the groups
// in order.  (One thread per stamp walked its 64 units in turn: 29 us, all latency.)
__global__ void __launch_bounds__(256) k_fc_epi(const float* __restrict__ part, uint32_t ldp, uint32_t n,
                                                const __nv_bfloat16* __restrict__ wb, __nv_bfloat16* a4g,
                                                float* __restrict__ logits) {
  __shared__ float dots[8][32];
  const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
  const uint32_t b = blockIdx.x * 32 + lane;
  float v[8], dot = 0.f;
  if (b < n) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int j = grp * 8 + k;
      float acc = part[(size_t)j * ldp + b];
#pragma unroll
      for (int sp = 1; sp < kFcSplit; ++sp) acc += part[((size_t)sp * kHid + j) * ldp + b];
      v[k] = acc;
    }
    uint32_t pk[4];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int j = grp * 8 + k;
      const __nv_bfloat16 a = __float2bfloat16_rn(fmaxf(v[k] + ld(wb + kBf1 + j), 0.f));
      pk[k / 2] = (k & 1) ? pk[k / 2] | ((uint32_t)__bfloat16_as_ushort(a) << 16) : (uint32_t)__bfloat16_as_ushort(a);
      dot = fmaf(__bfloat162float(a), ld(wb + kWf2 + j), dot);
    }
    if (a4g) *reinterpret_cast<uint4*>(a4g + (size_t)b * kHid + grp * 8) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
  }
  dots[grp][lane] = dot;
  __syncthreads();
  if (grp == 0 && b < n) {
    float s = dots[0][lane];
#pragma unroll
    for (int g = 1; g < 8; ++g) s += dots[g][lane];
    logits[b] = s + ld(wb + kBf2);
  }
}

// ---- loss, fc2 gradients, fc1 output deltas ------------------------------------

// Blocks of 128 stamps: per-stamp loss and d loss / d logit, the fc1 output deltas
// g4[b][j] = glogit[b] * w2[j] * (a4[b][j] > 0), and this block's sums for the fc2
// gradients and the loss: lpart[block][66] = fc2.w (64), fc2.b, loss.  k_fc1_sum
// adds the blocks in order.
constexpr int kLossStamps = 128, kLossOut = kHid + 2;

__global__ void __launch_bounds__(256) k_loss(const float* __restrict__ logits, const float* __restrict__ labels,
                                              const uint32_t* __restrict__ idx, uint32_t n,
                                              const __nv_bfloat16* __restrict__ a4g,
                                              const __nv_bfloat16* __restrict__ wb, float* __restrict__ g4,
                                              float* __restrict__ lpart) {
  __shared__ float gl[kLossStamps], red[256], redb[kLossStamps / 32], redl[kLossStamps / 32];
  const int t = threadIdx.x;
  const float inv_n = 1.f / (float)n;
  const uint32_t b0 = blockIdx.x * kLossStamps, nb = min((uint32_t)kLossStamps, n - b0);
  if (t < kLossStamps) {
    float l = 0.f, g = 0.f;
    if ((uint32_t)t < nb) {
      const uint32_t b = b0 + t;
      const float z = logits[b], y = labels[idx ? idx[b] : b];
      l = fmaxf(z, 0.f) - z * y + log1pf(expf(-fabsf(z)));
      g = (1.f / (1.f + expf(-z)) - y) * inv_n;
    }
    gl[t] = g;
    for (int o = 16; o > 0; o >>= 1) {
      l += __shfl_xor_sync(0xffffffffu, l, o);
      g += __shfl_xor_sync(0xffffffffu, g, o);
    }
    if ((t & 31) == 0) {
      redb[t >> 5] = g;
      redl[t >> 5] = l;
    }
  }
  __syncthreads();
  const int j = t & 63, part = t >> 6;
  const float w2 = ld(wb + kWf2 + j);
  float acc = 0.f;
#pragma unroll 8
  for (uint32_t r = part; r < nb; r += 4) {
    const size_t at = (size_t)(b0 + r) * kHid + j;
    const float a = ld(a4g + at), g = gl[r];
    acc = fmaf(g, a, acc);
    g4[at] = a > 0.f ? g * w2 : 0.f;
  }
  red[t] = acc;
  __syncthreads();
  float* out = lpart + (size_t)blockIdx.x * kLossOut;
  if (t < kHid) out[t] = ((red[t] + red[64 + t]) + red[128 + t]) + red[192 + t];
  if (t == 64) out[kHid] = ((redb[0] + redb[1]) + redb[2]) + redb[3];
  if (t == 65) out[kHid + 1] = ((redl[0] + redl[1]) + redl[2]) + redl[3];
}

// fc1.w[j][k] = sum_b g4[b][j] * a3[b][k];  fc1.b[j] = sum_b g4[b][j]; on the tensor
// cores: M = 128 columns k (a3), N = 3 x 64 (j at each of the three BF16 parts of g4,
// split_fp32: exact products, FP32 sums), K = 16 stamps per MMA, both operands
// MN-major straight from the row-major arrays.  Grid (21 column tiles, S): slice s
// adds the stamps [s n / S, (s + 1) n / S) in chunks of 64 through two stages and
// writes part[s][j][k] and its bias sums part[S * 64 * kF + s * 64 + j]; k_fc1_sum adds
// the slices in order.  (On the CUDA cores: 90 us for 4096 stamps, 65 for 512.)
constexpr int kDwThreads = 256, kDwChunk = 64, kDwCols = 128;
constexpr int kDwTiles = (kF + kDwCols - 1) / kDwCols;
constexpr int kDwA = (kDwCols / 8) * kDwChunk * 16, kDwB = 24 * kDwChunk * 16, kDwStage = kDwA + kDwB;
constexpr int kDwSmem = 2 * kDwStage + 32;

__global__ void __launch_bounds__(kDwThreads, 2) k_fc1_dw(const float* __restrict__ g4,
                                                          const __nv_bfloat16* __restrict__ a3g, uint32_t n,
                                                          float* __restrict__ part, uint32_t* __restrict__ status) {
  extern __shared__ __align__(1024) unsigned char smd[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(smd + 2 * kDwStage);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 2);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t S = gridDim.y, s = blockIdx.y;
  const uint32_t lo = (uint32_t)((uint64_t)n * s / S), hi = (uint32_t)((uint64_t)n * (s + 1) / S);
  const int k0 = blockIdx.x * kDwCols;
  if (warp == 0) tc::tmem_alloc(tslot, 256);
  if (tid == 0) {
    tc::mbar_init(bar, 1);
    tc::mbar_init(bar + 1, 1);
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tslot;
  const int jc = tid & 7;  // this thread's chunk of 8 hidden units
  float accb[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) accb[j] = 0.f;
  uint32_t ph = 0;  // bit st: parity of stage st's next wait
  bool ok = true;
  int l = 0;
  for (uint32_t c0 = lo; c0 < hi; c0 += kDwChunk, ++l) {
    const int st = l & 1;
    unsigned char* A = smd + st * kDwStage;
    unsigned char* B = A + kDwA;
    if (l >= 2) {
      ok = tc::mbar_wait(bar + st, (ph >> st) & 1u, 1u << 22);
      ph ^= 1u << st;
      if (__syncthreads_or(!ok)) {
        ok = false;
        break;
      }
    }
    for (int i = tid; i < (kDwCols / 8) * kDwChunk; i += kDwThreads) {
      const int c = i & 15, r = i >> 4;
      const bool in = c0 + r < hi && k0 + 8 * c < kF;
      tc::cp16(A + (c * kDwChunk + r) * 16, a3g + (in ? (size_t)(c0 + r) * kF + k0 + 8 * c : 0), in);
    }
    tc::cp_commit();
#pragma unroll
    for (int i = 0; i < kDwChunk * 8 / kDwThreads; ++i) {
      const int r = (tid + i * kDwThreads) >> 3;
      float4 v0 = make_float4(0.f, 0.f, 0.f, 0.f), v1 = v0;
      if (c0 + r < hi) {
        const float4* src = reinterpret_cast<const float4*>(g4 + (size_t)(c0 + r) * kHid + jc * 8);
        v0 = src[0];
        v1 = src[1];
      }
      const float v[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
      uint32_t pk[3][4];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        uint16_t p[3];
        tc::split_fp32(v[j], p[0], p[1], p[2]);
#pragma unroll
        for (int k = 0; k < 3; ++k) pk[k][j / 2] = (j & 1) ? pk[k][j / 2] | ((uint32_t)p[k] << 16) : (uint32_t)p[k];
        accb[j] += v[j];
      }
#pragma unroll
      for (int k = 0; k < 3; ++k)
        reinterpret_cast<uint4*>(B)[(k * 8 + jc) * kDwChunk + r] = make_uint4(pk[k][0], pk[k][1], pk[k][2], pk[k][3]);
    }
    tc::cp_wait<0>();
    tc::fence_smem_to_async();
    tc::fence_before_sync();
    __syncthreads();
    if (tid == 0) {
      tc::fence_after_sync();
      const uint32_t a0 = tc::smem_u32(A), b0 = tc::smem_u32(B);
      constexpr uint32_t id = tc::idesc_bf16_mn(128, 192);
#pragma unroll
      for (int k = 0; k < kDwChunk / 16; ++k)
        tc::mma_bf16(tmem, tc::smem_desc_strided(a0 + (uint32_t)(16 * k) * 16u, 128u, kDwChunk * 16u),
                     tc::smem_desc_strided(b0 + (uint32_t)(16 * k) * 16u, 128u, kDwChunk * 16u), id, (l | k) != 0);
      tc::commit(bar + st);
    }
  }
  for (int st = 0; st < 2 && ok; ++st)
    if (l > st) ok = tc::mbar_wait(bar + st, (ph >> st) & 1u, 1u << 22);
  if (__syncthreads_or(!ok)) ok = false;
  if (!ok) {
    if (tid == 0) atomicOr(status, 1u);
  } else {
    tc::fence_after_sync();
    const int q = warp & 3, h = warp >> 2;  // lane quadrant, half of the hidden units
    const int k = k0 + q * 32 + lane;
    float* pw = part + (size_t)s * kHid * kF;
#pragma unroll
    for (int jj = 0; jj < 32; jj += 16) {
      float v[3][16];
#pragma unroll
      for (int p = 0; p < 3; ++p)
        tc::ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(p * kHid + h * 32 + jj), v[p]);
      if (k < kF) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          pw[(size_t)(h * 32 + jj + j) * kF + k] = hi > lo ? (v[0][j] + v[1][j]) + v[2][j] : 0.f;
      }
    }
    if (blockIdx.x == 0) {
      float* red = reinterpret_cast<float*>(smd);  // [8 j][256]: the MMAs are done
#pragma unroll
      for (int j = 0; j < 8; ++j) red[j * kDwThreads + tid] = accb[j];
      __syncthreads();
      if (tid < kHid) {
        float v = 0.f;
        for (int r = 0; r < kDwThreads / 8; ++r) v += red[(tid & 7) * kDwThreads + r * 8 + (tid >> 3)];
        part[(size_t)S * kHid * kF + (size_t)s * kHid + tid] = v;
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_free(tmem, 256);
}

// grad[fc1.w] and grad[fc1.b]: the S slices of k_fc1_dw added in slice order; the
// last block adds k_loss's blocks: grad[fc2] and the mean loss.
__global__ void k_fc1_sum(const float* __restrict__ part, uint32_t S, const float* __restrict__ lpart, uint32_t n_loss,
                          uint32_t n, float* __restrict__ grad, float* __restrict__ loss) {
  if (blockIdx.x == gridDim.x - 1) {
    const uint32_t t = threadIdx.x;
    if (t >= kLossOut) return;
    float v = 0.f;
#pragma unroll 8
    for (uint32_t b = 0; b < n_loss; ++b) v += lpart[(size_t)b * kLossOut + t];
    if (t < kHid + 1)
      grad[(t < kHid ? kWf2 + t : kBf2)] = v;
    else
      *loss = v * (1.f / (float)n);
    return;
  }
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < (uint32_t)(kHid * kF)) {
    float v = 0.f;
#pragma unroll 4
    for (uint32_t s = 0; s < S; ++s) v += part[(size_t)s * kHid * kF + i];
    grad[kWf1 + i] = v;
  } else if (i < (uint32_t)(kHid * kF + kHid)) {
    const uint32_t j = i - kHid * kF;
    float v = 0.f;
    for (uint32_t s = 0; s < S; ++s) v += part[(size_t)S * kHid * kF + s * kHid + j];
    grad[kBf1 + j] = v;
  }
}

// g3[b][k] = (sum_j g4[b][j] * fc1.w[j][k]) * (a3[b][k] > 0), in FP32 with j in order.
// Block: 128 columns k x 64 stamps, 4 x 8 per thread: three 16-byte shared loads
// feed 32 multiply-adds (one column x 8 stamps took nine loads for eight: 76 us for
// 4096 stamps; the FP32 pipes need 17).
constexpr int kDxCols = 128, kDxStamps = 64;
constexpr int kDxSmem = kHid * (kDxCols + kDxStamps + 4) * 4;

__global__ void __launch_bounds__(256) k_fc1_dx(const float* __restrict__ g4,
                                                const __nv_bfloat16* __restrict__ wb,
                                                const __nv_bfloat16* __restrict__ a3g, uint32_t n,
                                                float* __restrict__ g3) {
  extern __shared__ __align__(16) float smx[];
  float* Ws = smx;                      // [64 j][128 k]
  float* Gs = smx + kHid * kDxCols;     // [64 j][64 stamps + 4]
  constexpr int kG = kDxStamps + 4;
  const int t = threadIdx.x, tx = t & 31, ty = t >> 5;
  const int k0 = blockIdx.x * kDxCols;
  const uint32_t b0 = blockIdx.y * kDxStamps;
  for (int i = t; i < kHid * kDxCols / 4; i += 256) {  // four weights at a time (kF is a multiple of 4)
    const int j = i / (kDxCols / 4), c = (i % (kDxCols / 4)) * 4;
    uint2 w = make_uint2(0, 0);
    if (k0 + c < kF) w = *reinterpret_cast<const uint2*>(wb + kWf1 + (size_t)j * kF + k0 + c);
    *reinterpret_cast<float4*>(Ws + j * kDxCols + c) =
        make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                    __uint_as_float(w.y & 0xffff0000u));
  }
  for (int i = t; i < kDxStamps * kHid; i += 256) {
    const uint32_t r = i / kHid, j = i % kHid;
    Gs[j * kG + r] = b0 + r < n ? g4[(size_t)(b0 + r) * kHid + j] : 0.f;
  }
  __syncthreads();
  float acc[8][4] = {};
#pragma unroll 4
  for (int j = 0; j < kHid; ++j) {
    const float4 w = *reinterpret_cast<const float4*>(Ws + j * kDxCols + 4 * tx);
    const float4 ga = *reinterpret_cast<const float4*>(Gs + j * kG + 8 * ty);
    const float4 gb = *reinterpret_cast<const float4*>(Gs + j * kG + 8 * ty + 4);
    const float g[8] = {ga.x, ga.y, ga.z, ga.w, gb.x, gb.y, gb.z, gb.w};
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      acc[s][0] = fmaf(g[s], w.x, acc[s][0]);
      acc[s][1] = fmaf(g[s], w.y, acc[s][1]);
      acc[s][2] = fmaf(g[s], w.z, acc[s][2]);
      acc[s][3] = fmaf(g[s], w.w, acc[s][3]);
    }
  }
  const int k = k0 + 4 * tx;
  if (k >= kF) return;
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const uint32_t b = b0 + 8 * ty + s;
    if (b >= n) break;
    const uint2 a = *reinterpret_cast<const uint2*>(a3g + (size_t)b * kF + k);
    auto on = [](uint32_t bits) { return bits != 0u && bits < 0x8000u; };  // a > 0
    *reinterpret_cast<float4*>(g3 + (size_t)b * kF + k) =
        make_float4(on(a.x & 0xffffu) ? acc[s][0] : 0.f, on(a.x >> 16) ? acc[s][1] : 0.f,
                    on(a.y & 0xffffu) ? acc[s][2] : 0.f, on(a.y >> 16) ? acc[s][3] : 0.f);
  }
}

// ---- conv backward on the tensor cores -------------------------------------------
//
// Per block (a fixed set of stamps, so gradients stay bit-reproducible), for a
// 32-channel layer with HI x HI inputs and HO x HO outputs:
//   dX[q][c] = sum_(tap, o) g[o][q - tap] * w[o][c][tap]
//   dW[o][c][tap] = sum_p g[o][p] * a[c][p + tap]
// Both are implicit GEMMs over buffers laid out as in the forward: [8-channel
// chunk][pixel row][8 channels], rows 16 bytes apart, pixel rows of HI columns.
//   g sits at row (y + 2) HI + x + 2 with zeros around it, so dX is the forward's
//   shifted-descriptor convolution with the taps reversed (K-major, M = 128 input
//   pixels a tile, N = 32 channels c, K = 16 channels o per MMA).
//   For dW the same buffers are read MN-major (channels contiguous): M = channels o,
//   N = 32 channels c, K = 16 pixels per MMA; a tap is again a shifted start of a.
// The deltas enter as two BF16 parts, hi + lo = the value cut to TF32's 11 bits
// (split_tf32), and weights and activations are BF16 values: products are exact
// and add up in FP32, as with kind::tf32, but operands need no im2col, whose
// building on the CUDA cores took nearly all of the time: with it 4096 stamps took
// 1.205 ms (HI = 13) and 0.804 ms (HI = 11), now 0.135 and 0.101.  hi and lo are 4 chunks each; a copy of both
// shifted by one pixel follows, so the 128 rows of one dW MMA are (hi, lo) at two
// neighbouring taps.  TMEM: dW 6 x 32 columns (per dy: taps 0 and 1, then tap 2 whose
// upper half is not used), dX 32 per tile; 256 in all, two CTAs per SM, so that one
// CTA's loads and epilogue overlap the other's MMAs.  The next stamp's values are
// fetched into registers while the MMAs run.  The masked dX goes to gout, bias
// gradients are FP32 sums of the uncut deltas.
constexpr int kBcThreads = 512;  // 16 warps: 4 TMEM lane quadrants x 4 eight-channel slices

template <int HI>
struct ConvBack {
  static constexpr int C = kCh, HO = HI - 2, P = HO * HO, Q = HI * HI, W = HI;
  static constexpr int MT = (Q + 127) / 128;               // dX tiles
  static constexpr int KD = (HO * W + 15) / 16 * 16;       // dW's K: g's pixels in rows of W
  static constexpr int OFF = 2 * W + 2;                    // row of g's first pixel
  static constexpr int RG = (MT * 128 + OFF + 7) / 8 * 8;  // rows of g: the last tile's last tap ends here
  static constexpr int RA = (KD + OFF + 7) / 8 * 8;        // rows of a
  static constexpr int kSmA = 16 * RG * 16;
  static constexpr int kSmW = kSmA + 4 * RA * 16;
  static constexpr int kSmBar = kSmW + 9 * C * C * 2;
  static constexpr int kSmem = kSmBar + 32;
  static constexpr int GI = (4 * P + kBcThreads - 1) / kBcThreads;  // (chunk, pixel) items per thread
  static constexpr int AI = (4 * Q + kBcThreads - 1) / kBcThreads;
  static_assert(OFF + KD + 1 <= RG && RA >= Q, "dW windows stay inside the buffers");
  static_assert(32 * 32 * 9 * 4 <= kSmA && 8 * kBcThreads * 4 <= kSmA, "the last sums fit g's buffer");
  static_assert(2 * kSmem <= 225 * 1024 && kSmA % 128 == 0 && kSmW % 128 == 0, "two CTAs per SM, operand alignment");
  static_assert(GI == 1, "a thread keeps one (chunk, pixel) of g: its bias sums");
};

template <int HI>
__global__ void __launch_bounds__(kBcThreads, 2) k_conv_back_tc(
    const float* __restrict__ gin, const __nv_bfloat16* __restrict__ ain, uint32_t n,
    const __nv_bfloat16* __restrict__ w, float* __restrict__ gout, float* __restrict__ partial,
    uint32_t* __restrict__ status) {
  using L = ConvBack<HI>;
  constexpr int C = L::C, HO = L::HO, P = L::P, Q = L::Q, W = L::W, RG = L::RG, RA = L::RA;
  extern __shared__ __align__(1024) unsigned char smb[];
  unsigned char* Ab = smb + L::kSmA;
  unsigned char* Wb = smb + L::kSmW;
  uint64_t* bar = reinterpret_cast<uint64_t*>(smb + L::kSmBar);  // dX done, dW done
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 2);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q4 = warp & 3, h = warp >> 2;
  if (warp == 0) tc::tmem_alloc(tslot, 256);
  if (tid == 0) {
    tc::mbar_init(bar, 1);
    tc::mbar_init(bar + 1, 1);
  }
  for (int i = tid; i < L::kSmW / 16; i += kBcThreads) reinterpret_cast<uint4*>(smb)[i] = make_uint4(0, 0, 0, 0);
  for (int i = tid; i < 9 * C * C; i += kBcThreads) {  // dX's B operand per tap: B_t[c][o] = w[o][c][t]
    const int o = i / (9 * C), c = (i / 9) % C, t = i % 9;
    *reinterpret_cast<__nv_bfloat16*>(Wb + t * C * C * 2 + tc::cm_offset(c, o, 4)) = w[i];
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tslot;
  const uint32_t g0 = tc::smem_u32(smb), a0 = tc::smem_u32(Ab), w0 = tc::smem_u32(Wb);
  const int g_chunk = tid / P, g_p = tid - g_chunk * P;
  const bool g_item = tid < 4 * P;
  const int g_row = L::OFF + (g_p / HO) * W + g_p % HO;
  float gv[8], accb[8];
  uint32_t av[L::AI][4];
#pragma unroll
  for (int j = 0; j < 8; ++j) gv[j] = accb[j] = 0.f;
  auto fetch = [&](uint32_t b) {
    if (b >= n) return;
    const float* g = gin + (size_t)b * C * P + g_chunk * 8 * P + g_p;
    if (g_item) {
#pragma unroll
      for (int j = 0; j < 8; ++j) gv[j] = g[j * P];
    }
    const uint16_t* a = reinterpret_cast<const uint16_t*>(ain) + (size_t)b * C * Q;
#pragma unroll
    for (int i = 0; i < L::AI; ++i) {
      const int it = tid + i * kBcThreads, chunk = it / Q, q = it - chunk * Q;
      if (it < 4 * Q) {
#pragma unroll
        for (int j = 0; j < 8; j += 2)
          av[i][j / 2] = (uint32_t)a[(chunk * 8 + j) * Q + q] | ((uint32_t)a[(chunk * 8 + j + 1) * Q + q] << 16);
      }
    }
  };
  fetch(blockIdx.x);
  uint32_t phase = 0, any = 0;
  bool ok = true;
  for (uint32_t b = blockIdx.x; b < n; b += gridDim.x) {
    if (g_item) {
      uint32_t hi[4], lo[4];
#pragma unroll
      for (int j = 0; j < 8; j += 2) {
        uint16_t h0, l0, h1, l1;
        tc::split_tf32(gv[j], h0, l0);
        tc::split_tf32(gv[j + 1], h1, l1);
        hi[j / 2] = (uint32_t)h0 | ((uint32_t)h1 << 16);
        lo[j / 2] = (uint32_t)l0 | ((uint32_t)l1 << 16);
        accb[j] += gv[j];
        accb[j + 1] += gv[j + 1];
      }
      const uint4 vh = make_uint4(hi[0], hi[1], hi[2], hi[3]), vl = make_uint4(lo[0], lo[1], lo[2], lo[3]);
      uint4* at = reinterpret_cast<uint4*>(smb) + g_chunk * RG + g_row;
      at[0] = vh;
      at[4 * RG] = vl;
      at[8 * RG + 1] = vh;   // the copy one pixel on
      at[12 * RG + 1] = vl;
    }
#pragma unroll
    for (int i = 0; i < L::AI; ++i) {
      const int it = tid + i * kBcThreads, chunk = it / Q, q = it - chunk * Q;
      if (it < 4 * Q)
        reinterpret_cast<uint4*>(Ab)[chunk * RA + q] = make_uint4(av[i][0], av[i][1], av[i][2], av[i][3]);
    }
    tc::fence_smem_to_async();
    tc::fence_before_sync();
    __syncthreads();
    if (tid == 0) {
      tc::fence_after_sync();
      constexpr uint32_t id_x = tc::idesc_bf16(128, 32), id_w = tc::idesc_bf16_mn(128, 32);
      for (int t = 0; t < L::MT; ++t)
        for (int tap = 0; tap < 9; ++tap) {
          const uint32_t shift = (uint32_t)((2 - tap / 3) * W + 2 - tap % 3) + (uint32_t)(t * 128);
#pragma unroll
          for (int k = 0; k < 4; ++k)  // hi, channels 0-15 and 16-31, then lo
            tc::mma_bf16(tmem + 192u + (uint32_t)(t * 32),
                         tc::smem_desc_strided(g0 + ((uint32_t)(2 * k * RG) + shift) * 16u, (uint32_t)(RG * 16), 128u),
                         tc::smem_desc(w0 + (uint32_t)(tap * C * C * 2 + 2 * (k & 1) * 128), 4), id_x, (tap | k) != 0);
        }
      tc::commit(bar);
      for (int blk = 0; blk < 6; ++blk) {  // taps (dy, 0) and (dy, 1) for blk = dy; (dy, 2) for blk = 3 + dy
        const uint32_t shift = (uint32_t)((blk % 3) * W + (blk < 3 ? 0 : 2));
        for (int k = 0; k < L::KD / 16; ++k)
          tc::mma_bf16(tmem + (uint32_t)(blk * 32),
                       tc::smem_desc_strided(g0 + (uint32_t)(L::OFF + 16 * k) * 16u, 128u, (uint32_t)(RG * 16)),
                       tc::smem_desc_strided(a0 + (shift + (uint32_t)(16 * k)) * 16u, 128u, (uint32_t)(RA * 16)), id_w,
                       any | (uint32_t)k);
      }
      tc::commit(bar + 1);
    }
    any = 1;
    fetch(b + gridDim.x);
    ok = tc::mbar_wait(bar, phase, 1u << 22);
    if (__syncthreads_or(!ok)) {
      ok = false;
      break;
    }
    tc::fence_after_sync();
    float* go = gout + (size_t)b * C * Q;
#pragma unroll
    for (int t = 0; t < L::MT; ++t) {
      float v[8];
      tc::ld8(tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(192 + t * 32 + h * 8), v);
      const int q = t * 128 + q4 * 32 + lane;
      if (q < Q) {  // mask by the input's ReLU
        const uint4 a = reinterpret_cast<const uint4*>(Ab)[h * RA + q];
        const uint32_t aw[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint32_t bits = (aw[j / 2] >> (16 * (j & 1))) & 0xffffu;
          go[(h * 8 + j) * Q + q] = bits != 0u && bits < 0x8000u ? v[j] : 0.f;
        }
      }
    }
    ok = tc::mbar_wait(bar + 1, phase, 1u << 22);
    phase ^= 1u;
    tc::fence_before_sync();
    if (__syncthreads_or(!ok)) {  // the buffers and dX's columns are free for the next stamp
      ok = false;
      break;
    }
    tc::fence_after_sync();
  }
  if (!ok && tid == 0) atomicOr(status, 1u);
  float* out = partial + (size_t)blockIdx.x * kPartialStride;  // [32 o][C][9], then [32] biases
  if (ok) {
    // dW: lanes 0-31 and 32-63 are hi and lo of output channel o at the block's first
    // tap, 64-95 and 96-127 at its second; both parts are added in shared memory
    tc::fence_after_sync();
    float* sum = reinterpret_cast<float*>(smb);
    for (int part = 0; part < 2; ++part) {
      if ((q4 & 1) == part) {
        for (int blk = 0; blk < (q4 < 2 ? 6 : 3); ++blk) {
          float v[8];
          tc::ld8(tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(blk * 32 + h * 8), v);
          const int tap = (blk % 3) * 3 + (blk < 3 ? q4 / 2 : 2);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            float* s = sum + (lane * C + h * 8 + j) * 9 + tap;
            *s = (part ? *s : 0.f) + v[j];
          }
        }
      }
      __syncthreads();
    }
    for (int i = tid; i < C * C * 9; i += kBcThreads) out[i] = any ? sum[i] : 0.f;
    __syncthreads();
    // biases: 16 threads per channel add its pixels' sums
#pragma unroll
    for (int j = 0; j < 8; ++j) sum[j * kBcThreads + tid] = accb[j];
    __syncthreads();
    const int o = tid >> 4;
    float s = 0.f;
    for (int p = tid & 15; p < P; p += 16) s += sum[(o & 7) * kBcThreads + (o >> 3) * P + p];
#pragma unroll
    for (int x = 8; x > 0; x >>= 1) s += __shfl_xor_sync(0xffffffffu, s, x);
    if ((tid & 15) == 0) out[C * C * 9 + o] = s;
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_free(tmem, 256);
}

// ---- conv1 weight gradient ---------------------------------------------------------
//
// dW[o][c][tap] = sum_p g1[o][p] x[c][p + tap] over 9 input channels of 15 x 15
// counts, per block as above.  The deltas enter in full, as three BF16 parts (hi,
// mid, lo: split_fp32), the inputs are BF16 values, so every product is exact and
// adds up in FP32 as on the CUDA cores before (4096 stamps: 0.203 ms, now 0.098).  Both
// operands MN-major: M = (3 parts x 32 channels o, 32 rows unused), N = 16 (9 channels
// c), K = 16 pixels of rows of 15 columns; a tap is a shifted start of x.
constexpr int kC1K = 208;                    // 13 rows of 15 columns, padded to 16
constexpr int kC1RG = kC1K, kC1RX = 240;     // rows: x to 207 + 2 * 15 + 2
constexpr int kC1SmX = 16 * kC1RG * 16;      // chunks 12..15 of g's buffer are never written
constexpr int kC1SmBar = kC1SmX + 2 * kC1RX * 16;
constexpr int kC1Smem = kC1SmBar + 16;
constexpr int kC1Items = (4 * kH1 * kH1 + kBcThreads - 1) / kBcThreads;  // (chunk, pixel) items per thread
static_assert(kC1RX >= kC1K + 2 * kS + 2 && kC1RX >= kS * kS && 2 * kC1Smem <= 225 * 1024, "conv1 windows");
static_assert(kCh * kQ * 9 * 4 <= kC1SmX && 2 * 8 * kBcThreads * 4 <= kC1SmX, "the last sums fit g's buffer");

__global__ void __launch_bounds__(kBcThreads, 2) k_conv1_dw_tc(const float* __restrict__ gin,
                                                               const uint16_t* __restrict__ stamps,
                                                               const uint32_t* __restrict__ idx, uint32_t n,
                                                               float* __restrict__ partial,
                                                               uint32_t* __restrict__ status) {
  constexpr int C = kCh, P = kH1 * kH1, Q = kS * kS;
  extern __shared__ __align__(1024) unsigned char smb[];
  uint16_t* xs = reinterpret_cast<uint16_t*>(smb + kC1SmX);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smb + kC1SmBar);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q4 = warp & 3, h = warp >> 2;
  if (warp == 0) tc::tmem_alloc(tslot, 256);  // 9 taps x 16 columns
  if (tid == 0) tc::mbar_init(bar, 1);
  for (int i = tid; i < kC1SmBar / 16; i += kBcThreads) reinterpret_cast<uint4*>(smb)[i] = make_uint4(0, 0, 0, 0);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tslot, g0 = tc::smem_u32(smb), x0 = tc::smem_u32(smb + kC1SmX);
  constexpr int kPer = (kQ * Q + kBcThreads - 1) / kBcThreads;
  float gv[kC1Items][8], accb[kC1Items][8];
  uint16_t xv[kPer];
#pragma unroll
  for (int i = 0; i < kC1Items; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) gv[i][j] = accb[i][j] = 0.f;
  auto fetch = [&](uint32_t b) {
    if (b >= n) return;
#pragma unroll
    for (int i = 0; i < kC1Items; ++i) {
      const int it = tid + i * kBcThreads, chunk = it / P, p = it - chunk * P;
      if (it < 4 * P) {
#pragma unroll
        for (int j = 0; j < 8; ++j) gv[i][j] = gin[(size_t)b * C * P + (chunk * 8 + j) * P + p];
      }
    }
    const uint16_t* st = stamps + (size_t)(idx ? idx[b] : b) * kQ * Q;
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
      const int i = tid + r * kBcThreads;
      xv[r] = i < kQ * Q ? st[i] : (uint16_t)0;
    }
  };
  fetch(blockIdx.x);
  uint32_t phase = 0, any = 0;
  bool ok = true;
  for (uint32_t b = blockIdx.x; b < n; b += gridDim.x) {
#pragma unroll
    for (int i = 0; i < kC1Items; ++i) {
      const int it = tid + i * kBcThreads, chunk = it / P, p = it - chunk * P;
      if (it < 4 * P) {
        uint32_t part[3][4];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          uint16_t v[3];
          tc::split_fp32(gv[i][j], v[0], v[1], v[2]);
#pragma unroll
          for (int k = 0; k < 3; ++k)
            part[k][j / 2] = (j & 1) ? part[k][j / 2] | ((uint32_t)v[k] << 16) : (uint32_t)v[k];
          accb[i][j] += gv[i][j];
        }
        uint4* at = reinterpret_cast<uint4*>(smb) + chunk * kC1RG + (p / kH1) * kS + p % kH1;
#pragma unroll
        for (int k = 0; k < 3; ++k) at[4 * k * kC1RG] = make_uint4(part[k][0], part[k][1], part[k][2], part[k][3]);
      }
    }
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
      const int i = tid + r * kBcThreads;
      if (i < kQ * Q) {
        const int c = i / Q, p = i - c * Q;
        xs[((c >> 3) * kC1RX + p) * 8 + (c & 7)] = __bfloat16_as_ushort(__float2bfloat16_rn((float)xv[r] * 0.0625f));
      }
    }
    tc::fence_smem_to_async();
    tc::fence_before_sync();
    __syncthreads();
    if (tid == 0) {
      tc::fence_after_sync();
      constexpr uint32_t id = tc::idesc_bf16_mn(128, 16);
      for (int tap = 0; tap < 9; ++tap)
        for (int k = 0; k < kC1K / 16; ++k)
          tc::mma_bf16(tmem + (uint32_t)(tap * 16),
                       tc::smem_desc_strided(g0 + (uint32_t)(16 * k) * 16u, 128u, (uint32_t)(kC1RG * 16)),
                       tc::smem_desc_strided(x0 + (uint32_t)((tap / 3) * kS + tap % 3 + 16 * k) * 16u, 128u,
                                             (uint32_t)(kC1RX * 16)),
                       id, any | (uint32_t)k);
      tc::commit(bar);
    }
    any = 1;
    fetch(b + gridDim.x);
    ok = tc::mbar_wait(bar, phase, 1u << 22);
    phase ^= 1u;
    if (__syncthreads_or(!ok)) {
      ok = false;
      break;
    }
  }
  if (!ok && tid == 0) atomicOr(status, 1u);
  float* out = partial + (size_t)blockIdx.x * kPartialStride;  // [32 o][9 c][9], then [32] biases
  if (ok) {
    tc::fence_after_sync();
    float* sum = reinterpret_cast<float*>(smb);
    for (int part = 0; part < 3; ++part) {  // lanes 32 part + o
      if (q4 == part && h < 2) {
        for (int tap = 0; tap < 9; ++tap) {
          float v[8];
          tc::ld8(tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(tap * 16 + h * 8), v);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int c = h * 8 + j;
            if (c < kQ) {
              float* s = sum + (lane * kQ + c) * 9 + tap;
              *s = (part ? *s : 0.f) + v[j];
            }
          }
        }
      }
      __syncthreads();
    }
    for (int i = tid; i < C * kQ * 9; i += kBcThreads) out[i] = sum[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kC1Items; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) sum[j * (kC1Items * kBcThreads) + tid + i * kBcThreads] = accb[i][j];
    __syncthreads();
    const int o = tid >> 4;
    float s = 0.f;
    for (int p = tid & 15; p < P; p += 16) s += sum[(o & 7) * (kC1Items * kBcThreads) + (o >> 3) * P + p];
#pragma unroll
    for (int x = 8; x > 0; x >>= 1) s += __shfl_xor_sync(0xffffffffu, s, x);
    if ((tid & 15) == 0) out[C * kQ * 9 + o] = s;
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_free(tmem, 256);
}

// The conv layers' gradients from their blocks' partial sums (weights, then
// biases: rows of kPartialStride per block, layer l at l * kBackBlocks rows).  Blocks
// of 32 elements x 8 groups of rows: a row's 32 elements are read together, each
// group adds its rows in order, the groups are added in order.  (A warp per element,
// its lanes over the rows, read a sector for every value: 19 us a layer.)
__global__ void __launch_bounds__(256) k_reduce_partials(const float* __restrict__ partial, int n_blocks,
                                                         float* __restrict__ grad) {
  __shared__ float red[8][32];
  const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5, l = blockIdx.y;  // l: conv1, conv2, conv3
  const int nw = l == 0 ? kCh * kQ * 9 : kCh * kCh * 9, i = blockIdx.x * 32 + lane;
  const float* p = partial + (size_t)l * kBackBlocks * kPartialStride + i;
  float s = 0.f;
  if (i < nw + kCh) {
    const int r0 = n_blocks * grp / 8, r1 = n_blocks * (grp + 1) / 8;
#pragma unroll 8
    for (int r = r0; r < r1; ++r) s += p[(size_t)r * kPartialStride];
  }
  red[grp][lane] = s;
  __syncthreads();
  if (grp == 0 && i < nw + kCh) {
#pragma unroll
    for (int g = 1; g < 8; ++g) s += red[g][lane];
    const int w_off = l == 0 ? kW1 : l == 1 ? kW2 : kW3, b_off = l == 0 ? kB1 : l == 1 ? kB2 : kB3;
    grad[i < nw ? w_off + i : b_off + (i - nw)] = s;
  }
}

// ---- parameters --------------------------------------------------------------

__global__ void k_cast(const float* __restrict__ master, __nv_bfloat16* __restrict__ wb) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kNParams) return;
  wb[i] = __float2bfloat16_rn(master[i]);
}

// Adam (Kingma & Ba 2015) on the FP32 master values; refreshes the BF16 copies.
__global__ void k_adam(float* __restrict__ master, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ grad, float lr, float beta1, float beta2, float eps,
                       float bc1, float bc2, __nv_bfloat16* __restrict__ wb) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kNParams) return;
  const float g = grad[i];
  const float mi = beta1 * m[i] + (1.f - beta1) * g;
  const float vi = beta2 * v[i] + (1.f - beta2) * g * g;
  m[i] = mi;
  v[i] = vi;
  const float p = master[i] - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
  master[i] = p;
  wb[i] = __float2bfloat16_rn(p);
}

// ---- host side -----------------------------------------------------------------

// Shared-memory limits of the kernels on the current device (they are the device's own,
// so every vetter sets them on its device).
cudaError_t set_attrs() {
  cudaError_t e = cudaFuncSetAttribute(k_conv_fwd_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_fc_fwd_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kFcTcSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_conv_back_tc<kH2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             ConvBack<kH2>::kSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_conv_back_tc<kH1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             ConvBack<kH1>::kSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_fc1_dx, cudaFuncAttributeMaxDynamicSharedMemorySize, kDxSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_fc1_dw, cudaFuncAttributeMaxDynamicSharedMemorySize, kDwSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_conv1_dw_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kC1Smem);
  return e;
}

// Forward of n <= max_batch stamps; with keep, stores the activations training needs.
cudaError_t forward(sas_vet* vt, const uint16_t* stamps, const uint32_t* idx, uint32_t n, bool keep,
                    float* logits, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int blocks = (int)std::min<uint32_t>(n, (uint32_t)vt->sms);
  k_conv_fwd_tc<<<blocks, kTcThreads, kTcSmem, s>>>(stamps, idx, n, vt->wb, keep ? vt->a1 : nullptr,
                                                   keep ? vt->a2 : nullptr, vt->a3, vt->status);
  const uint32_t tiles = (n + kFcTcRows - 1) / kFcTcRows, ldp = tiles * kFcTcRows;
  k_fc_fwd_tc<<<dim3(tiles, kFcSplit), kFcTcThreads, kFcTcSmem, s>>>(vt->a3, n, vt->wb, vt->fcpart, ldp,
                                                                     vt->status);
  k_fc_epi<<<(n + 31) / 32, 256, 0, s>>>(vt->fcpart, ldp, n, vt->wb, keep ? vt->a4 : nullptr, logits);
  note_launch();
  note_launch(2);
  return cudaGetLastError();
}

cudaError_t gradients(sas_vet* vt, const uint16_t* stamps, const float* labels, const uint32_t* idx,
                      uint32_t n, float* grad, cudaStream_t s) {
  cudaError_t e = forward(vt, stamps, idx, n, true, vt->logits, s);
  if (e != cudaSuccess) return e;
  const uint32_t n_loss = (n + kLossStamps - 1) / kLossStamps;
  k_loss<<<n_loss, 256, 0, s>>>(vt->logits, labels, idx, n, vt->a4, vt->wb, vt->g4, vt->lpart);
  // stamp slices: enough blocks for two per SM, at least one chunk each
  const uint32_t S = std::max<uint32_t>(1, std::min<uint32_t>(kFc1Slices, n / kDwChunk));
  k_fc1_dw<<<dim3(kDwTiles, S), kDwThreads, kDwSmem, s>>>(vt->g4, vt->a3, n, vt->partial, vt->status);
  k_fc1_sum<<<(kHid * kF + kHid + 255) / 256 + 1, 256, 0, s>>>(vt->partial, S, vt->lpart, n_loss, n, grad, vt->loss);
  k_fc1_dx<<<dim3((kF + kDxCols - 1) / kDxCols, (n + kDxStamps - 1) / kDxStamps), 256, kDxSmem, s>>>(
      vt->g4, vt->wb, vt->a3, n, vt->g3);
  const int nb = (int)std::min<uint32_t>(n, kBackBlocks);
  const size_t per = (size_t)kBackBlocks * kPartialStride;
  k_conv_back_tc<kH2><<<nb, kBcThreads, ConvBack<kH2>::kSmem, s>>>(vt->g3, vt->a2, n, vt->wb + kW3, vt->g2,
                                                                 vt->partial + 2 * per, vt->status);
  k_conv_back_tc<kH1><<<nb, kBcThreads, ConvBack<kH1>::kSmem, s>>>(vt->g2, vt->a1, n, vt->wb + kW2, vt->g1,
                                                                 vt->partial + per, vt->status);
  k_conv1_dw_tc<<<nb, kBcThreads, kC1Smem, s>>>(vt->g1, stamps, idx, n, vt->partial, vt->status);
  k_reduce_partials<<<dim3((kCh * kCh * 9 + kCh + 31) / 32, 3), 256, 0, s>>>(vt->partial, nb, grad);
  note_launch(8);
  return cudaGetLastError();
}

cudaError_t adam(sas_vet* vt, const float* grad, float lr, cudaStream_t s) {
  vt->step += 1;
  const double bc1 = 1.0 - std::pow((double)vt->beta1, (double)vt->step);
  const double bc2 = 1.0 - std::pow((double)vt->beta2, (double)vt->step);
  k_adam<<<(kNParams + 255) / 256, 256, 0, s>>>(vt->master, vt->m, vt->v, grad, lr, vt->beta1, vt->beta2,
                                               vt->eps, (float)bc1, (float)bc2, vt->wb);
  note_launch();
  return cudaGetLastError();
}

}  // namespace vet

cudaError_t vet_forward_all(sas_vet* vt, const uint16_t* stamps, uint64_t n, float* logits, cudaStream_t s) {
  for (uint64_t b0 = 0; b0 < n; b0 += vt->max_batch) {
    const uint32_t nb = (uint32_t)std::min<uint64_t>(vt->max_batch, n - b0);
    cudaError_t e = vet::forward(vt, stamps + b0 * 9 * 225, nullptr, nb, false, logits + b0, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

int vet_device(const sas_vet* vt) { return vt->device; }

}  // namespace sas

// ---- C ABI -----------------------------------------------------------------------

using namespace sas;

namespace {

struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    cudaGetDevice(&prev);
    if (prev != dev) cudaSetDevice(dev);
  }
  ~DeviceGuard() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};

int cuda_fail(cudaError_t e, const char* what) {
  return set_errorf(SAS_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

void free_vet(sas_vet* vt) {
  void* ptrs[] = {vt->master, vt->m, vt->v, vt->grad, vt->wb, vt->a1, vt->a2, vt->a3,
                  vt->a4, vt->logits, vt->lpart, vt->g4, vt->g3, vt->g2, vt->g1, vt->partial, vt->loss,
                  vt->status, vt->fcpart};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  delete vt;
}

}  // namespace

extern "C" {

uint64_t sas_vet_num_params(void) { return (uint64_t)vet::kNParams; }

int sas_vet_create(int device, uint32_t max_batch, sas_vet** out) {
  if (!out) return set_error(SAS_ERR_ARG, "sas_vet_create: out is NULL");
  *out = nullptr;
  if (max_batch == 0 || max_batch > SAS_VET_MAX_BATCH)
    return set_errorf(SAS_ERR_ARG, "sas_vet_create: max_batch must be 1..%u", (unsigned)SAS_VET_MAX_BATCH);
  DeviceGuard guard(device);
  int sms = 0;
  cudaError_t ae = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  if (ae == cudaSuccess) ae = vet::set_attrs();
  if (ae != cudaSuccess) return cuda_fail(ae, "sas_vet_create");
  sas_vet* vt = new sas_vet();
  std::memset(vt, 0, sizeof(*vt));
  vt->device = device;
  vt->sms = sms;
  vt->max_batch = max_batch;
  vt->beta1 = 0.9f;
  vt->beta2 = 0.999f;
  vt->eps = 1e-8f;
  const size_t B = max_batch, N = vet::kNParams;
  struct Req {
    void** p;
    size_t bytes;
  } reqs[] = {
      {(void**)&vt->master, N * 4}, {(void**)&vt->m, N * 4}, {(void**)&vt->v, N * 4},
      {(void**)&vt->grad, N * 4}, {(void**)&vt->wb, N * 2},
      {(void**)&vt->a1, B * vet::kCh * vet::kH1 * vet::kH1 * 2}, {(void**)&vt->a2, B * vet::kCh * vet::kH2 * vet::kH2 * 2},
      {(void**)&vt->a3, B * vet::kF * 2}, {(void**)&vt->a4, B * vet::kHid * 2}, {(void**)&vt->logits, B * 4},
      {(void**)&vt->lpart, (B + vet::kLossStamps - 1) / vet::kLossStamps * vet::kLossOut * 4},
      {(void**)&vt->g4, B * vet::kHid * 4}, {(void**)&vt->g3, B * vet::kF * 4},
      {(void**)&vt->g2, B * vet::kCh * vet::kH2 * vet::kH2 * 4}, {(void**)&vt->g1, B * vet::kCh * vet::kH1 * vet::kH1 * 4},
      {(void**)&vt->partial, (size_t)3 * vet::kBackBlocks * vet::kPartialStride * 4}, {(void**)&vt->loss, 4},
      {(void**)&vt->status, 4},
      {(void**)&vt->fcpart, (size_t)vet::kFcSplit * vet::kHid * ((B + 127) / 128 * 128) * 4},
  };
  for (auto& r : reqs) {
    if (cudaError_t e = cudaMalloc(r.p, r.bytes); e != cudaSuccess) {
      free_vet(vt);
      return cuda_fail(e, "sas_vet_create: cudaMalloc");
    }
  }
  cudaMemset(vt->status, 0, 4);
  cudaMemset(vt->master, 0, N * 4);
  cudaMemset(vt->m, 0, N * 4);
  cudaMemset(vt->v, 0, N * 4);
  vet::k_cast<<<(vet::kNParams + 255) / 256, 256>>>(vt->master, vt->wb);
  note_launch();
  if (cudaError_t e = cudaDeviceSynchronize(); e != cudaSuccess) {
    free_vet(vt);
    return cuda_fail(e, "sas_vet_create");
  }
  *out = vt;
  return SAS_OK;
}

int sas_vet_destroy(sas_vet* vt) {
  if (!vt) return SAS_OK;
  DeviceGuard guard(vt->device);
  cudaDeviceSynchronize();
  free_vet(vt);
  return SAS_OK;
}

int sas_vet_check(sas_vet* vt) {
  if (!vt) return set_error(SAS_ERR_ARG, "sas_vet_check: NULL vetter");
  DeviceGuard guard(vt->device);
  uint32_t st = 0;
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = cudaMemcpy(&st, vt->status, 4, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && st) e = cudaMemset(vt->status, 0, 4);
  if (e != cudaSuccess) return cuda_fail(e, "sas_vet_check");
  if (st) return set_error(SAS_ERR_TIMEOUT, "sas_vet_check: a tensor-core wait gave up; logits are incomplete");
  return SAS_OK;
}

int sas_vet_set_adam(sas_vet* vt, float beta1, float beta2, float eps) {
  if (!vt) return set_error(SAS_ERR_ARG, "sas_vet_set_adam: NULL vetter");
  if (!(beta1 >= 0.f && beta1 < 1.f && beta2 >= 0.f && beta2 < 1.f && eps > 0.f))
    return set_error(SAS_ERR_ARG, "sas_vet_set_adam: need 0 <= beta < 1 and eps > 0");
  vt->beta1 = beta1;
  vt->beta2 = beta2;
  vt->eps = eps;
  return SAS_OK;
}

int sas_vet_set_state(sas_vet* vt, const float* params, const float* m, const float* v, uint64_t step) {
  if (!vt || !params) return set_error(SAS_ERR_ARG, "sas_vet_set_state: NULL argument");
  if ((m == nullptr) != (v == nullptr))
    return set_error(SAS_ERR_ARG, "sas_vet_set_state: give both Adam moments or neither");
  DeviceGuard guard(vt->device);
  const size_t bytes = (size_t)vet::kNParams * 4;
  cudaError_t e = cudaMemcpy(vt->master, params, bytes, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = m ? cudaMemcpy(vt->m, m, bytes, cudaMemcpyHostToDevice) : cudaMemset(vt->m, 0, bytes);
  if (e == cudaSuccess) e = v ? cudaMemcpy(vt->v, v, bytes, cudaMemcpyHostToDevice) : cudaMemset(vt->v, 0, bytes);
  if (e != cudaSuccess) return cuda_fail(e, "sas_vet_set_state");
  vt->step = m ? step : 0;
  vet::k_cast<<<(vet::kNParams + 255) / 256, 256>>>(vt->master, vt->wb);
  note_launch();
  e = cudaDeviceSynchronize();
  return e == cudaSuccess ? SAS_OK : cuda_fail(e, "sas_vet_set_state");
}

int sas_vet_get_state(const sas_vet* vt, float* params, float* m, float* v, uint64_t* step) {
  if (!vt) return set_error(SAS_ERR_ARG, "sas_vet_get_state: NULL vetter");
  DeviceGuard guard(vt->device);
  const size_t bytes = (size_t)vet::kNParams * 4;
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess && params) e = cudaMemcpy(params, vt->master, bytes, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && m) e = cudaMemcpy(m, vt->m, bytes, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && v) e = cudaMemcpy(v, vt->v, bytes, cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "sas_vet_get_state");
  if (step) *step = vt->step;
  return SAS_OK;
}

int sas_vet_get_bf16(const sas_vet* vt, uint16_t* out) {
  if (!vt || !out) return set_error(SAS_ERR_ARG, "sas_vet_get_bf16: NULL argument");
  DeviceGuard guard(vt->device);
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = cudaMemcpy(out, vt->wb, (size_t)vet::kNParams * 2, cudaMemcpyDeviceToHost);
  return e == cudaSuccess ? SAS_OK : cuda_fail(e, "sas_vet_get_bf16");
}

int sas_vet_get_activations(const sas_vet* vt, uint32_t layer, uint64_t n, uint16_t* out) {
  if (!vt || (n && !out)) return set_error(SAS_ERR_ARG, "sas_vet_get_activations: NULL argument");
  if (layer < 1 || layer > 4) return set_error(SAS_ERR_ARG, "sas_vet_get_activations: layer must be 1..4");
  if (n > vt->max_batch) return set_error(SAS_ERR_ARG, "sas_vet_get_activations: n exceeds the vetter's batch");
  const size_t per = layer == 1 ? (size_t)vet::kCh * vet::kH1 * vet::kH1
                   : layer == 2 ? (size_t)vet::kCh * vet::kH2 * vet::kH2
                   : layer == 3 ? (size_t)vet::kF : (size_t)vet::kHid;
  const __nv_bfloat16* src = layer == 1 ? vt->a1 : layer == 2 ? vt->a2 : layer == 3 ? vt->a3 : vt->a4;
  DeviceGuard guard(vt->device);
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess && n) e = cudaMemcpy(out, src, n * per * 2, cudaMemcpyDeviceToHost);
  return e == cudaSuccess ? SAS_OK : cuda_fail(e, "sas_vet_get_activations");
}

int sas_vet_forward(sas_vet* vt, const uint16_t* stamps, const uint32_t* index, uint64_t n, float* logits,
                    void* stream) {
  if (!vt) return set_error(SAS_ERR_ARG, "sas_vet_forward: NULL vetter");
  if (n && (!stamps || !logits)) return set_error(SAS_ERR_ARG, "sas_vet_forward: NULL buffer");
  DeviceGuard guard(vt->device);
  cudaStream_t s = (cudaStream_t)stream;
  for (uint64_t b0 = 0; b0 < n; b0 += vt->max_batch) {
    const uint32_t nb = (uint32_t)std::min<uint64_t>(vt->max_batch, n - b0);
    const uint16_t* st = index ? stamps : stamps + b0 * 9 * 225;
    if (cudaError_t e = vet::forward(vt, st, index ? index + b0 : nullptr, nb, false, logits + b0, s);
        e != cudaSuccess)
      return cuda_fail(e, "sas_vet_forward");
  }
  return SAS_OK;
}

int sas_vet_gradients(sas_vet* vt, const uint16_t* stamps, const float* labels, const uint32_t* index,
                      uint32_t n, float* grad, float* loss, void* stream) {
  if (!vt) return set_error(SAS_ERR_ARG, "sas_vet_gradients: NULL vetter");
  if (n == 0 || n > vt->max_batch)
    return set_errorf(SAS_ERR_ARG, "sas_vet_gradients: n must be 1..%u", vt->max_batch);
  if (!stamps || !labels || !grad) return set_error(SAS_ERR_ARG, "sas_vet_gradients: NULL buffer");
  DeviceGuard guard(vt->device);
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = vet::gradients(vt, stamps, labels, index, n, grad, s);
  if (e == cudaSuccess && loss) e = cudaMemcpyAsync(loss, vt->loss, 4, cudaMemcpyDeviceToDevice, s);
  return e == cudaSuccess ? SAS_OK : cuda_fail(e, "sas_vet_gradients");
}

int sas_vet_apply_gradients(sas_vet* vt, const float* grad, float lr, void* stream) {
  if (!vt || !grad) return set_error(SAS_ERR_ARG, "sas_vet_apply_gradients: NULL argument");
  if (!(lr >= 0.f)) return set_error(SAS_ERR_ARG, "sas_vet_apply_gradients: lr must be >= 0");
  DeviceGuard guard(vt->device);
  cudaError_t e = vet::adam(vt, grad, lr, (cudaStream_t)stream);
  return e == cudaSuccess ? SAS_OK : cuda_fail(e, "sas_vet_apply_gradients");
}

int sas_vet_train_step(sas_vet* vt, const uint16_t* stamps, const float* labels, const uint32_t* index,
                       uint32_t n, float lr, float* loss, void* stream) {
  if (!vt) return set_error(SAS_ERR_ARG, "sas_vet_train_step: NULL vetter");
  if (n == 0 || n > vt->max_batch)
    return set_errorf(SAS_ERR_ARG, "sas_vet_train_step: n must be 1..%u", vt->max_batch);
  if (!stamps || !labels) return set_error(SAS_ERR_ARG, "sas_vet_train_step: NULL buffer");
  if (!(lr >= 0.f)) return set_error(SAS_ERR_ARG, "sas_vet_train_step: lr must be >= 0");
  DeviceGuard guard(vt->device);
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = vet::gradients(vt, stamps, labels, index, n, vt->grad, s);
  if (e == cudaSuccess) e = vet::adam(vt, vt->grad, lr, s);
  if (e == cudaSuccess && loss) e = cudaMemcpyAsync(loss, vt->loss, 4, cudaMemcpyDeviceToDevice, s);
  return e == cudaSuccess ? SAS_OK : cuda_fail(e, "sas_vet_train_step");
}

}  // extern "C"
