// C ABI of the shift-and-stack library: validation, planning and the launch
// sequence of one search (Sec. 2.1 steps 1-3).
#include <algorithm>
#include <atomic>
#include <chrono>
#include <cstdlib>
#include <cmath>
#include <cstdarg>
#include <cstddef>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "sas_internal.cuh"

using namespace sas;

struct sas_grid {
  sas_grid_desc d;
  // emissions of the previous search on this grid -- super-bins of a one-level search,
  // windows of a two-level one: they size the next emission list of the same
  // kind so that repeated searches do not need an exact rerun
  std::atomic<uint32_t> emit_hint{0}, window_hint{0};
};

struct sas_result {
  int device;
  void* d_mem;        // one allocation: the bucketed catalog and tables below
  void* d_out;        // one allocation: candidates and ids (null in a cluster list)
  sas_candidate* d_cands;
  uint32_t* d_ids;
  sas_result_info info;
  // The search's bucketed catalog, per-epoch counts and shift tables, kept so
  // that stamps can be cut from the same search (sas_stamps).
  Det* d_dets;
  uint32_t* d_boff;
  uint32_t* d_ecount;
  int32_t* d_sxt;
  int32_t* d_syt;
  int64_t* d_dt;      // per-epoch time minus t0, ticks
  SearchGeom g;
  CoarseGeom cg;
  uint64_t n_det;     // catalog size (detection ids are < n_det)
  uint32_t n_min;     // the search's threshold (the score threshold when weighted)
  int complete;       // every cell >= n_min is in the list (no top-K cut)
  int weighted;       // counts are weighted scores
  int two_levels;     // found by the window search
};

namespace {
thread_local std::string g_err;
}  // namespace

namespace sas {
std::atomic<unsigned long long> g_launches{0};
void note_launch(uint32_t k) { g_launches.fetch_add(k, std::memory_order_relaxed); }

int set_errorf(int code, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  g_err = buf;
  return code;
}
}  // namespace sas

namespace {

template <typename... Args>
int fail(int code, const char* fmt, Args... args) {
  return set_errorf(code, fmt, args...);
}

int cuda_fail(cudaError_t e, const char* where) {
  return fail(e == cudaErrorMemoryAllocation ? SAS_ERR_OOM : SAS_ERR_CUDA, "%s: %s", where,
              cudaGetErrorString(e));
}

// Stream-ordered scratch, released when the search returns.
struct Scratch {
  cudaStream_t s;
  std::vector<void*> ptrs;
  explicit Scratch(cudaStream_t st) : s(st) {}
  ~Scratch() {
    for (void* p : ptrs) cudaFreeAsync(p, s);
  }
  template <typename T>
  cudaError_t alloc(T** p, size_t count) {
    void* q = nullptr;
    cudaError_t e = cudaMallocAsync(&q, std::max<size_t>(count, 1) * sizeof(T), s);
    if (e != cudaSuccess) return e;
    ptrs.push_back(q);
    *p = static_cast<T*>(q);
    return cudaSuccess;
  }
};

// Several arrays in one allocation: add() them, allocate `size` bytes, place() them.
struct Arena {
  size_t size = 0;
  struct Part {
    void** p;
    size_t at;
  };
  std::vector<Part> parts;
  template <typename T>
  void add(T** p, size_t count) {
    parts.push_back({(void**)p, size});
    size += (std::max<size_t>(count, 1) * sizeof(T) + 255) & ~size_t(255);
  }
  void place(char* base) {
    for (const Part& q : parts) *q.p = base + q.at;
  }
};

// Windows that a two-level search lists (1 GB); more leave the field to the one-level search.
constexpr uint32_t kMaxWindows = 1u << 26;

// What the kernels of a search report, in one block so that one copy reads it.
struct Counters {
  uint32_t flags, n_emit, n_valid, n_long;  // n_long: windows that the long pass counts
  unsigned long long pairs, tile, raw, balance, pairs1, n_ids;  // pairs1: of the window search's first level
  long long t0;
};

bool fits_i32(int64_t v) { return v >= INT32_MIN && v <= INT32_MAX; }

// Opt-in host-side tracing (environment variable SAS_TRACE=1): microseconds
// since the start of the call at each phase boundary, on stderr.
struct Tracer {
  bool on;
  std::chrono::steady_clock::time_point t0;
  Tracer() : on(std::getenv("SAS_TRACE") != nullptr), t0(std::chrono::steady_clock::now()) {}
  void mark(const char* what) const {
    if (!on) return;
    const double us = std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now() - t0).count();
    std::fprintf(stderr, "[sas] %9.1f us  %s\n", us, what);
  }
};

}  // namespace

namespace sas {
bool result_two_levels(const sas_result* r) { return r->two_levels != 0; }

CandView result_view(const sas_result* r) {
  CandView v;
  v.cands = r->d_cands;
  v.n = r->info.n_candidates;
  v.g = r->g;
  v.cg = r->cg;
  v.dets = r->d_dets;
  v.boff = r->d_boff;
  v.ecount = r->d_ecount;
  v.sxt = r->d_sxt;
  v.syt = r->d_syt;
  v.ids = r->d_ids;
  v.n_det = r->n_det;
  return v;
}
}  // namespace sas

extern "C" {

const char* sas_version(void) { return "sas-gb300 0.1 (sm_103a)"; }
int sas_abi_version(void) { return SAS_ABI_VERSION; }
uint64_t sas_kernel_launches(void) { return sas::g_launches.load(); }
const char* sas_last_error(void) { return g_err.c_str(); }

int sas_create_grid(const sas_grid_desc* desc, sas_grid** out) {
  if (!desc || !out) return fail(SAS_ERR_ARG, "null argument");
  const sas_grid_desc& d = *desc;
  if (d.nvx < 1 || d.nvy < 1 || d.nbx < 1 || d.nby < 1 || d.bin < 1)
    return fail(SAS_ERR_ARG, "lattice and domain sizes and the bin must be >= 1");
  if (d.speed_min < 0 || d.speed_max < d.speed_min)
    return fail(SAS_ERR_ARG, "need 0 <= speed_min <= speed_max");
  if ((uint64_t)d.nvx * d.nvy >= ((uint64_t)1 << 31))
    return fail(SAS_ERR_RANGE, "nvx*nvy must be < 2^31");
  if (std::llabs((int64_t)d.x_min) >= kLimDomain || std::llabs((int64_t)d.y_min) >= kLimDomain)
    return fail(SAS_ERR_RANGE, "|x_min|, |y_min| must be < 2^28");
  if ((int64_t)d.nbx * d.bin >= kLimDomain || (int64_t)d.nby * d.bin >= kLimDomain)
    return fail(SAS_ERR_RANGE, "nbx*bin and nby*bin must be < 2^28");
  if (!fits_i32((int64_t)d.vx0 + (int64_t)(d.nvx - 1) * d.dvx) ||
      !fits_i32((int64_t)d.vy0 + (int64_t)(d.nvy - 1) * d.dvy))
    return fail(SAS_ERR_RANGE, "lattice velocities must fit in int32");
  sas_grid* g = new (std::nothrow) sas_grid;
  if (!g) return fail(SAS_ERR_OOM, "host allocation");
  g->d = d;
  g->emit_hint.store(0);
  g->window_hint.store(0);
  *out = g;
  return SAS_OK;
}

void sas_destroy_grid(sas_grid* grid) { delete grid; }

int sas_grid_get_desc(const sas_grid* grid, sas_grid_desc* desc) {
  if (!grid || !desc) return fail(SAS_ERR_ARG, "null argument");
  *desc = grid->d;
  return SAS_OK;
}

namespace {

// The search (Sec. 2.1 steps 1-3); with weights (one uint8 per detection, in
// host or device memory like the catalog) cells are scored by the sum over
// epochs of their largest weight and n_min is the score threshold.
// window_bits: the least counter width of a window search (sas_hier.cu), 0 for none; a
// field that turns out not to fit it is searched again with wider counters or without.
int stack_impl(const sas_grid* grid, const sas_catalog* cat, const uint8_t* weights, uint32_t n_min,
               const sas_opts* opts, void* stream, sas_result** out, int window_bits = 8) {
  if (!grid || !cat || !out) return fail(SAS_ERR_ARG, "null argument");
  const Tracer tr;
  const sas_grid_desc& d = grid->d;
  const uint32_t E = cat->n_epochs;
  const uint64_t n = cat->n;
  if (n_min < 1) return fail(SAS_ERR_ARG, "n_min must be >= 1");
  if (E < 1 || E > SAS_MAX_EPOCHS) return fail(SAS_ERR_RANGE, "n_epochs must be in [1, %d]", SAS_MAX_EPOCHS);
  if (!cat->t) return fail(SAS_ERR_ARG, "null epoch time table");
  if (cat->ticks_per_hour <= 0) return fail(SAS_ERR_ARG, "ticks_per_hour must be > 0");
  if (n >= ((uint64_t)1 << 31)) return fail(SAS_ERR_RANGE, "n must be < 2^31");
  if (n > 0 && (!cat->x || !cat->y || !cat->epoch)) return fail(SAS_ERR_ARG, "null catalog array");
  sas_opts o{};
  if (opts) o = *opts;
  const uint64_t nv = (uint64_t)d.nvx * d.nvy;
  uint64_t v_begin = o.v_begin, v_end = o.v_end;
  if (v_begin == 0 && v_end == 0) v_end = nv;
  if (v_begin > v_end || v_end > nv) return fail(SAS_ERR_ARG, "bad lattice index range");
  int64_t tmin = cat->t[0], tmax = cat->t[0];
  for (uint32_t e = 1; e < E; ++e) {
    tmin = std::min(tmin, cat->t[e]);
    tmax = std::max(tmax, cat->t[e]);
  }
  if ((__int128)tmax - tmin >= ((__int128)1 << 32)) return fail(SAS_ERR_RANGE, "time span must be < 2^32 ticks");
  const int64_t tph = cat->ticks_per_hour;

  int dev = 0;
  cudaError_t ce = cudaGetDevice(&dev);
  if (ce != cudaSuccess) return cuda_fail(ce, "cudaGetDevice");
  DevInfo di;
  if (int rc = device_info(dev, &di)) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  if (n_min > (1u << 31)) return fail(SAS_ERR_ARG, "n_min must be <= 2^31");
  if (o.n_low > n_min) return fail(SAS_ERR_ARG, "n_low %u is above n_min %u", o.n_low, n_min);
  if ((o.n_low || o.peaks_only) && weights)
    return fail(SAS_ERR_ARG, "n_low and peaks_only are not supported by the weighted search");
  if (o.peaks_only > 1) return fail(SAS_ERR_ARG, "peaks_only must be 0 or 1");
  const uint32_t n_low = o.n_low ? o.n_low : n_min;

  sas_result* res = new (std::nothrow) sas_result;
  if (!res) return fail(SAS_ERR_OOM, "host allocation");
  memset(res, 0, sizeof(*res));
  res->device = dev;
  res->n_det = n;
  res->n_min = n_min;
  res->info.n_low = n_low;
  res->info.peaks_only = o.peaks_only;

  if (n == 0 || v_begin == v_end) {
    res->info.t0 = 0;
    res->complete = 1;
    *out = res;
    return SAS_OK;
  }

  res->weighted = weights != nullptr;
  // The largest weight sizes the super-bins and the mean one the windows.
  double mean_weight = 0;
  int sb_auto = 0;
  if (weights && o.superbin == 0) {
    unsigned long long st[2] = {0, 0};
    if (cat->on_device) {
      unsigned long long* d_st = nullptr;
      ce = cudaMallocAsync((void**)&d_st, 16, s);
      if (ce == cudaSuccess) {
        ce = launch_weight_stats(weights, n, d_st, s);
        if (ce == cudaSuccess) ce = cudaMemcpyAsync(st, d_st, 16, cudaMemcpyDeviceToHost, s);
        if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
        cudaFreeAsync(d_st, s);
      }
      if (ce != cudaSuccess) {
        delete res;
        return cuda_fail(ce, "weights");
      }
    } else {
      for (uint64_t i = 0; i < n; ++i) {
        st[0] = std::max<unsigned long long>(st[0], weights[i]);
        st[1] += weights[i];
      }
    }
    const uint32_t wmax = std::max((uint32_t)st[0], 1u);
    mean_weight = std::max((double)st[1] / (double)n, 0.01);
    // the super-bin heuristic models unit increments: give it the distinct-epoch
    // count that a score of n_min needs at the largest weight
    sb_auto = choose_superbin(d, n, (n_min + wmax - 1) / wmax, v_end - v_begin);
  }
  sas_opts op = o;  // with the super-bin side that the weights ask for
  if (sb_auto) op.superbin = (uint32_t)sb_auto;

  FieldPlan plan;
  if (int rc = plan_field(d, n, E, cat->t, tph, n_min, v_begin, v_end, op, di, &plan)) {
    delete res;
    return rc;
  }
  // A caller that sets tile sizes gets the one-level kernel with those tiles.
  WindowPlan wplan;
  const bool use_win = window_bits && n_low == n_min && !o.peaks_only && !o.tile_kx && !o.tile_ky && !o.tile_bx &&
                       !o.tile_by && !o.counter_bits && !o.coarse_bins && !o.superbin && !o.velocity_block &&
                       plan_windows(d, n, n_min, mean_weight, v_begin, v_end, di, plan, &wplan, window_bits);
  int again = -1;  // the window search gave up: run again with these window_bits
  const CoarseGeom& cg = use_win ? wplan.cg : plan.cg;
  const uint64_t nb = use_win ? wplan.nb : plan.nb;
  const SearchGeom& g = plan.g;
  tr.mark("planned");

  cudaEvent_t ev0, ev1, evs0, evs1, evc0, evc1;
  cudaEventCreate(&ev0); cudaEventCreate(&ev1); cudaEventCreate(&evs0); cudaEventCreate(&evs1);
  cudaEventCreate(&evc0); cudaEventCreate(&evc1);
  struct EvGuard {
    cudaEvent_t e[6];
    ~EvGuard() { for (cudaEvent_t x : e) cudaEventDestroy(x); }
  } evg{{ev0, ev1, evs0, evs1, evc0, evc1}};
  cudaEventRecord(ev0, s);

  int rc = SAS_OK;
  {
    Scratch sc(s);
#define CK(expr, where)                          \
  do {                                           \
    cudaError_t e_ = (expr);                     \
    if (e_ != cudaSuccess) {                     \
      rc = cuda_fail(e_, where);                 \
      goto done;                                 \
    }                                            \
  } while (0)
    const int32_t* dx = cat->x;
    const int32_t* dy = cat->y;
    const uint16_t* dep = cat->epoch;
    const uint8_t* d_w = weights;
    const bool host = !cat->on_device;
    std::atomic<uint32_t>& last_emit = const_cast<sas_grid*>(grid)->*(use_win ? &sas_grid::window_hint : &sas_grid::emit_hint);
    const uint32_t hint = last_emit.load(std::memory_order_relaxed);
    uint32_t emit_cap = (uint32_t)std::min<uint64_t>(
        std::max<uint64_t>({use_win ? (uint64_t)wplan.list_cap : std::max<uint64_t>((uint64_t)1 << 16, 2 * n),
                            (uint64_t)hint + hint / 4 + 1024}), (uint64_t)1 << 26);
    uint32_t key_cap = use_win ? 1u << 17 : 0;
    const size_t npts = use_win && wplan.masked ? ((size_t)d.nvx + 1) * ((size_t)d.nvy + 1) : 0;
    const size_t nK = use_win ? (size_t)wplan.g.nvx * wplan.g.nvy : 0;
    Counters h{};
    uint32_t n_out = 0;
    StackArgs sa{};
    WindowArgs wa{};
    Key* sorted = nullptr;
    unsigned long long *d_idoff = nullptr, *d_scan64 = nullptr;
    uint32_t* d_ids_tmp = nullptr;

    // Two allocations up to the stack kernel: scratch, and what the result keeps.
    Counters* d_cnt = nullptr;
    int32_t *hx = nullptr, *hy = nullptr;
    uint16_t* hep = nullptr;
    uint8_t* hw = nullptr;
    int64_t* d_t = nullptr;
    uint32_t *d_bcount = nullptr, *d_cursor = nullptr, *d_bof = nullptr, *d_scan = nullptr;
    uint32_t *d_ecount = nullptr, *d_boff = nullptr;  // kept by the result, as are the next three
    Det* d_dets = nullptr;
    int32_t *d_sxt = nullptr, *d_syt = nullptr;
    Emit* d_emits = nullptr;
    Key* d_keys = nullptr;
    // Reads the counters back after the stack stage; the input errors of a search.
    auto read_counters = [&]() -> cudaError_t {
      cudaError_t e = cudaMemcpyAsync(&h, d_cnt, sizeof(h), cudaMemcpyDeviceToHost, s);
      return e == cudaSuccess ? cudaStreamSynchronize(s) : e;
    };
    auto input_error = [&]() -> int {
      if (h.flags & kFlagEpoch) return fail(SAS_ERR_RANGE, "an epoch index is >= n_epochs");
      if (h.flags & kFlagPos) return fail(SAS_ERR_RANGE, "a detection has |x| or |y| >= 2^29");
      if (h.flags & kFlagShift) return fail(SAS_ERR_RANGE, "a shift |v*(t-t0)/TPH| >= 2^28");
      if (h.flags & kFlagInternal) return fail(SAS_ERR_INTERNAL, "stack kernel invariant");
      return SAS_OK;
    };
    Arena scratch, keep;
    scratch.add(&d_cnt, 1);  // the counters and the bucket counts start at zero: one memset
    // nb grid buckets plus one overflow bucket (detections outside the grid)
    scratch.add(&d_bcount, nb + 1);
    const size_t zeroed = scratch.size;
    scratch.add(&d_t, E);
    scratch.add(&d_cursor, nb + 1);
    scratch.add(&d_scan, scan_scratch_elems(nb + 1));
    scratch.add(&d_bof, n);
    if (host) {
      scratch.add(&hx, n);
      scratch.add(&hy, n);
      scratch.add(&hep, n);
      if (weights) scratch.add(&hw, n);
    }
    scratch.add(&d_emits, emit_cap);
    if (use_win) {
      scratch.add(&d_keys, key_cap);
      scratch.add(&wa.sXt, (size_t)wplan.g.nvx * E);
      scratch.add(&wa.sYt, (size_t)wplan.g.nvy * E);
      scratch.add(&wa.mx, d.nvx);
      scratch.add(&wa.my, d.nvy);
      if (wplan.masked) {
        scratch.add(&wa.vact, nK);
        scratch.add(&wa.vsum, npts);
      }
    }
    keep.add(&res->d_ecount, E);
    keep.add(&res->d_dets, n);
    keep.add(&res->d_boff, nb + 2);
    keep.add(&res->d_sxt, (size_t)d.nvx * E);
    keep.add(&res->d_syt, (size_t)d.nvy * E);
    keep.add(&res->d_dt, E);
    {
      char* base = nullptr;
      CK(sc.alloc(&base, scratch.size), "alloc scratch");
      scratch.place(base);
      CK(cudaMallocAsync(&res->d_mem, keep.size, s), "alloc result");
      keep.place((char*)res->d_mem);
      CK(cudaMemsetAsync(base, 0, zeroed, s), "memset");
    }
    d_ecount = res->d_ecount;
    d_boff = res->d_boff;
    d_dets = res->d_dets;
    d_sxt = res->d_sxt;
    d_syt = res->d_syt;
    res->g = g;
    res->cg = cg;
    CK(cudaMemsetAsync(d_ecount, 0, E * 4, s), "memset");
    if (host) {
      CK(cudaMemcpyAsync(hx, cat->x, n * 4, cudaMemcpyHostToDevice, s), "copy x");
      CK(cudaMemcpyAsync(hy, cat->y, n * 4, cudaMemcpyHostToDevice, s), "copy y");
      CK(cudaMemcpyAsync(hep, cat->epoch, n * 2, cudaMemcpyHostToDevice, s), "copy epoch");
      dx = hx; dy = hy; dep = hep;
      if (weights) {
        CK(cudaMemcpyAsync(hw, weights, n, cudaMemcpyHostToDevice, s), "copy weights");
        d_w = hw;
      }
    }
    CK(cudaMemcpyAsync(d_t, cat->t, E * 8, cudaMemcpyHostToDevice, s), "copy t");
    tr.mark("allocated");

    // a1-a3: ingest and validate, bucket, reference epoch, shift tables
    CK(launch_ingest(dx, dy, dep, n, E, cg, d_bcount, d_ecount, d_bof, &d_cnt->flags, s), "ingest");
    CK(launch_scan_u32(d_bcount, d_boff, nb + 1, d_scan, s, d_cursor), "bucket scan");
    CK(launch_scatter(dx, dy, dep, n, d_bof, d_cursor, d_dets, s), "scatter");
    CK(launch_shift_tables(g, d_t, d_ecount, res->d_dt, (int64_t*)&d_cnt->t0, d_sxt, d_syt, &d_cnt->flags, s), "shift tables");
    tr.mark("prep launched");

    sa.w = d_w;
    sa.dets = d_dets;
    sa.boff = d_boff;
    sa.ecount = d_ecount;
    sa.n_emit = &d_cnt->n_emit;
    sa.balance = &d_cnt->balance;
    sa.flags = &d_cnt->flags;
    sa.tile_counter = &d_cnt->tile;

    if (use_win) {  // a4-a7 in two levels: windows of groups of velocities, then their bins
      const TileCfg& tc = wplan.tc;
      wa.gx = wplan.gx;
      wa.gy = wplan.gy;
      wa.win = wplan.win;
      wa.unit = wplan.unit;
      wa.g = g;
      wa.cgm = wplan.g;
      wa.cg = cg;
      wa.dets = d_dets;
      wa.boff = d_boff;
      wa.ecount = d_ecount;
      wa.dt = res->d_dt;
      wa.sxt = d_sxt;
      wa.syt = d_syt;
      wa.wts = d_w;
      wa.n_windows = &d_cnt->n_emit;
      wa.balance = &d_cnt->balance;
      wa.n_min = n_min;
      wa.n_valid = &d_cnt->n_valid;
      wa.raw_total = &d_cnt->raw;
      wa.n_pairs = &d_cnt->pairs;
      wa.flags = &d_cnt->flags;
      CK(stack_set_smem_attr_windows(tc.kx, tc.ky, tc.cb, tc.smem), "smem attribute");
      fill_window_args(wplan, n_min, (uint32_t)(v_begin / d.nvx), (uint32_t)((v_end - 1) / d.nvx), &sa);
      sa.vact = wa.vact;
      sa.sxt = wa.sXt;
      sa.syt = wa.sYt;
      sa.n_pairs = &d_cnt->pairs1;
      cudaEventRecord(evs0, s);
      CK(launch_window_tables(wa, s), "group tables");
      CK(launch_window_pairs(wa, dx, dy, dep, n, s), "pair count");
      wa.n_long = &d_cnt->n_long;
      for (bool level1 = true;;) {
        if (level1) {
          wa.windows = sa.emits = d_emits;
          wa.list_cap = sa.emit_cap = emit_cap;
          CK(launch_stack_windows(sa, (int)std::min<uint64_t>((uint64_t)di.sms, std::max<uint64_t>(sa.n_tiles, 1)), s),
             "window kernel");
          level1 = false;
        }
        wa.keys = d_keys;
        wa.key_cap = key_cap;
        CK(launch_window_cells(wa, di.sms, s), "window cells");
        if (wa.n_queue) CK(launch_window_long(wa, di.sms, s), "long windows");
        cudaEventRecord(evs1, s);
        CK(read_counters(), "stack sync");
        tr.mark("windows done");
        if ((rc = input_error())) goto done;
        const bool full = (h.flags & kFlagEmitCap) || h.n_emit > emit_cap, wrapped = h.balance != 0;
        if (wrapped || (h.flags & kFlagWindow) || (full && (h.n_emit <= emit_cap || h.n_emit > kMaxWindows))) {
          again = wrapped && wplan.tc.cb == 8 ? 16 : 0;
          rc = SAS_ERR_INTERNAL;
          goto done;
        }
        if (full) {  // level 1 again with room for what it found
          emit_cap = h.n_emit;
          CK(sc.alloc(&d_emits, emit_cap), "alloc windows");
          CK(cudaMemsetAsync(d_cnt, 0, offsetof(Counters, pairs), s), "memset");
          CK(cudaMemsetAsync(&d_cnt->tile, 0, offsetof(Counters, n_ids) - offsetof(Counters, tile), s), "memset");
          level1 = true;
          continue;
        }
        if (h.n_long != wa.n_queue) {  // long windows, known now
          wa.n_queue = h.n_long;
          CK(sc.alloc(&wa.queue, wa.n_queue), "alloc long windows");
          CK(cudaMemsetAsync(wa.n_long, 0, 4, s), "memset");
          CK(launch_window_queue(wa, di.sms, s), "long window queue");
          CK(launch_window_long(wa, di.sms, s), "long windows");
          cudaEventRecord(evs1, s);
          CK(read_counters(), "long windows sync");
          if (h.flags & kFlagWindow) {
            again = 0;
            rc = SAS_ERR_INTERNAL;
            goto done;
          }
        }
        if (h.n_valid <= key_cap) break;
        key_cap = h.n_valid;
        if (key_cap >= (1u << 30)) { rc = fail(SAS_ERR_OOM, "too many candidate bins; raise n_min"); goto done; }
        CK(sc.alloc(&d_keys, key_cap), "alloc keys");
        CK(cudaMemsetAsync(&d_cnt->n_valid, 0, 4, s), "memset");
        CK(cudaMemsetAsync(wa.n_long, 0, 4, s), "memset");
        CK(cudaMemsetAsync(&d_cnt->raw, 0, 8, s), "memset");
      }
      cudaEventRecord(evc0, s);
    }

    // a4-a6: the stack kernel; reruns (exact) with wider counters if one wrapped
    // or with a longer emission list if it overflowed.
    for (int attempt = 0; !use_win; ++attempt) {
      const TileCfg& tc = plan.tc;
      fill_stack_args(plan, n_min, n_low, o.peaks_only, &sa);
      CK(stack_set_smem_attr(tc.kx, tc.ky, tc.cb, tc.smem, sa.select != kSelectAll), "smem attribute");
      sa.sxt = d_sxt;
      sa.syt = d_syt;
      sa.emits = d_emits;
      sa.emit_cap = emit_cap;
      sa.n_pairs = &d_cnt->pairs;
      if (attempt > 0) {  // all but t0 starts again
        CK(cudaMemsetAsync(d_cnt, 0, offsetof(Counters, t0), s), "memset");
      }
      const int grid_sz = (int)std::min<uint64_t>((uint64_t)di.sms, std::max<uint64_t>(sa.n_tiles, 1));
      cudaEventRecord(evs0, s);
      tr.mark("stack configured");
      CK(launch_stack(sa, grid_sz, s), "stack kernel");
      cudaEventRecord(evs1, s);
      tr.mark("stack launched");
      CK(read_counters(), "stack sync");
      tr.mark("stack done");
      if ((rc = input_error())) goto done;
      if (attempt >= 4) { rc = fail(SAS_ERR_INTERNAL, "stack kernel did not converge"); goto done; }
      if ((h.flags & kFlagCounter) || h.balance != 0) {  // a counter wrapped
        if (int r2 = replan_wider(d, n, n_min, op, di, &plan)) { rc = r2; goto done; }
        continue;
      }
      if (h.n_emit > emit_cap || (h.flags & kFlagEmitCap)) {
        if (h.n_emit >= (1u << 28)) {
          rc = fail(SAS_ERR_OOM, "more than 2^28 cells reach the threshold; raise n_min");
          goto done;
        }
        emit_cap = h.n_emit + h.n_emit / 4 + 1024;
        CK(sc.alloc(&d_emits, emit_cap), "alloc emissions");
        continue;
      }
      // a5/a7: exact distinct and raw counts of every bin of the emitted super-bins
      const uint64_t n_keys = (uint64_t)h.n_emit * plan.tc.s * plan.tc.s;
      if (n_keys >= (1ull << 31)) { rc = fail(SAS_ERR_OOM, "too many candidate bins; raise n_min"); goto done; }
      CK(sc.alloc(&d_keys, n_keys), "alloc keys");
      cudaEventRecord(evc0, s);
      CK(launch_cell_count(d_emits, h.n_emit, plan.tc.s, g, cg, d_dets, d_boff, d_ecount, d_sxt,
                           d_syt, n_min, sa.n_low, d_keys, &d_cnt->n_valid, &d_cnt->raw, d_w, s), "cell count");
      if (h.n_emit) CK(read_counters(), "count sync");
      tr.mark("counts done");
      break;
    }
    {
      last_emit.store(h.n_emit, std::memory_order_relaxed);
      // a8: total order of the valid keys; a7: candidates, contributing ids
      const uint32_t n_emit = h.n_emit, n_valid = h.n_valid;
      n_out = n_valid;
      if (o.max_candidates > 0 && n_out > o.max_candidates) n_out = (uint32_t)o.max_candidates;
      const uint64_t id_cap = std::max<uint64_t>(h.raw, 1);
      uint32_t n_pad = 1;
      while (n_pad < n_valid) n_pad <<= 1;
      Arena post, mine;
      if (!sort_in_place(n_valid)) post.add(&sorted, n_valid > kSortMerge ? n_pad : n_valid);
      post.add(&d_idoff, (size_t)n_out + 1);
      post.add(&d_scan64, candidates_scratch_elems(n_out));
      post.add(&d_ids_tmp, id_cap);
      mine.add(&res->d_cands, n_out);
      mine.add(&res->d_ids, id_cap);
      {
        char* base = nullptr;
        CK(sc.alloc(&base, post.size), "alloc ordering");
        post.place(base);
        CK(cudaMallocAsync(&res->d_out, mine.size, s), "alloc result candidates");
        mine.place((char*)res->d_out);
      }
      if (!sorted) sorted = d_keys;
      CK(launch_sort(d_keys, n_valid, sorted, s), "sort");
      cudaEventRecord(evc1, s);
      CK(launch_candidates(sorted, n_out, d_idoff, d_scan64, res->d_cands, &d_cnt->n_ids, s), "candidates");
      CK(launch_gather_ids(sorted, n_out, d_idoff, g, cg, d_dets, d_boff, d_ecount, d_sxt, d_syt,
                           d_ids_tmp, res->d_ids, &d_cnt->flags, s), "gather ids");
      cudaEventRecord(ev1, s);
      CK(read_counters(), "final sync");
      tr.mark("ids done");
      if (h.flags & kFlagInternal) { rc = fail(SAS_ERR_INTERNAL, "id gather invariant"); goto done; }
      const unsigned long long n_ids = h.n_ids;
      res->info.n_candidates = n_out;
      res->complete = n_out == n_valid;
      res->two_levels = use_win;
      res->info.n_ids = n_ids;
      res->info.n_pairs = h.pairs;
      res->info.n_emitted = n_emit;
      res->info.t0 = h.t0;
      res->info.counter_bits = (uint32_t)(use_win ? wplan.tc.cb : plan.tc.cb);
      res->info.tile_kx = (uint32_t)plan.tc.kx;
      res->info.tile_ky = (uint32_t)plan.tc.ky;
      res->info.tile_bx = (uint32_t)plan.tc.tx;
      res->info.tile_by = (uint32_t)plan.tc.ty;
      res->info.superbin = (uint32_t)plan.tc.s;
      res->info.vblock_x = (uint32_t)plan.tc.bvx;
      res->info.vblock_y = (uint32_t)plan.tc.bvy;
      res->info.staged_cap = (uint32_t)plan.tc.scap;
      cudaEventElapsedTime(&res->info.ms_stack, evs0, evs1);
      cudaEventElapsedTime(&res->info.ms_total, ev0, ev1);
      cudaEventElapsedTime(&res->info.ms_count, evc0, evc1);
      cudaEventElapsedTime(&res->info.ms_ids, evc1, ev1);
      cudaEventElapsedTime(&res->info.ms_prep, ev0, evs0);
    }
  done:;
#undef CK
  }
  if (rc != SAS_OK) {
    for (void* p : {res->d_mem, res->d_out})
      if (p) cudaFreeAsync(p, s);
    cudaStreamSynchronize(s);
    delete res;
    return again >= 0 ? stack_impl(grid, cat, weights, n_min, opts, stream, out, again) : rc;
  }
  *out = res;
  return SAS_OK;
}

}  // namespace

int sas_stack(const sas_grid* grid, const sas_catalog* cat, uint32_t n_min, const sas_opts* opts,
              void* stream, sas_result** out) {
  return stack_impl(grid, cat, nullptr, n_min, opts, stream, out);
}

int sas_stack_weighted(const sas_grid* grid, const sas_catalog* cat, const uint8_t* weights, uint32_t s_min,
                       const sas_opts* opts, void* stream, sas_result** out) {
  if (!weights && cat && cat->n) return fail(SAS_ERR_ARG, "null weights");
  return stack_impl(grid, cat, weights ? weights : (const uint8_t*)"", s_min, opts, stream, out);
}

int sas_result_get_info(const sas_result* r, sas_result_info* info) {
  if (!r || !info) return fail(SAS_ERR_ARG, "null argument");
  *info = r->info;
  return SAS_OK;
}

int sas_candidates(const sas_result* r, sas_candidate* out, uint64_t cap, uint64_t* n_total,
                   uint32_t* ids, uint64_t ids_cap, uint64_t* n_ids_total, int on_device) {
  if (!r) return fail(SAS_ERR_ARG, "null result");
  const uint64_t nc = r->info.n_candidates, ni = r->info.n_ids;
  if (n_total) *n_total = nc;
  if (n_ids_total) *n_ids_total = ni;
  const uint64_t c1 = std::min(cap, nc), i1 = std::min(ids_cap, ni);
  const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  if (c1 && !out) return fail(SAS_ERR_ARG, "null candidate buffer");
  if (i1 && !ids) return fail(SAS_ERR_ARG, "null id buffer");
  // both copies on the legacy default stream (the search completed before it
  // returned), then one wait
  if (c1) {
    cudaError_t e = cudaMemcpyAsync(out, r->d_cands, c1 * sizeof(sas_candidate), kind, 0);
    if (e != cudaSuccess) return cuda_fail(e, "copy candidates");
  }
  if (i1) {
    cudaError_t e = cudaMemcpyAsync(ids, r->d_ids, i1 * sizeof(uint32_t), kind, 0);
    if (e != cudaSuccess) return cuda_fail(e, "copy ids");
  }
  if (c1 || i1) {
    cudaError_t e = cudaStreamSynchronize(0);
    if (e != cudaSuccess) return cuda_fail(e, "copy candidates");
  }
  if (cap < nc || ids_cap < ni)
    return fail(SAS_ERR_OVERFLOW, "buffers too small: need %llu candidates and %llu ids",
                (unsigned long long)nc, (unsigned long long)ni);
  return SAS_OK;
}

int sas_stamps(const sas_result* r, uint64_t first, uint64_t count, uint16_t* out, void* stream) {
  if (!r) return fail(SAS_ERR_ARG, "null result");
  if (!r->d_dets && count) return fail(SAS_ERR_ARG, "this result keeps no catalog (a cluster list)");
  const uint64_t nc = r->info.n_candidates;
  if (first > nc || count > nc - first)
    return fail(SAS_ERR_ARG, "candidates [%llu, %llu) outside the result's %llu", (unsigned long long)first,
                (unsigned long long)(first + count), (unsigned long long)nc);
  if (count == 0) return SAS_OK;
  if (!out) return fail(SAS_ERR_ARG, "null stamp buffer");
  cudaError_t e = launch_stamps(result_view(r), nullptr, first, count, out, (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e, "stamps");
  return SAS_OK;
}

int sas_stamps_indexed(const sas_result* r, const uint32_t* idx, uint64_t count, uint16_t* out,
                       void* stream) {
  if (!r) return fail(SAS_ERR_ARG, "null result");
  if (!r->d_dets && count) return fail(SAS_ERR_ARG, "this result keeps no catalog (a cluster list)");
  if (count == 0) return SAS_OK;
  if (!idx || !out) return fail(SAS_ERR_ARG, "null index or stamp buffer");
  cudaError_t e = launch_stamps(result_view(r), idx, 0, count, out, (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e, "stamps");
  return SAS_OK;
}

int sas_peel(const sas_result* r, uint32_t n_min, uint32_t max_clusters, uint32_t flags, void* stream,
             sas_result** out) {
  if (!r || !out) return fail(SAS_ERR_ARG, "null argument");
  if (!r->d_dets && r->info.n_candidates)
    return fail(SAS_ERR_ARG, "cluster finding needs a search result (this one is a cluster list)");
  if (n_min < r->n_min || n_min == 0)
    return fail(SAS_ERR_ARG, "n_min %u is below the search's threshold %u (cells under it are not in the list)",
                n_min, r->n_min);
  if (!r->complete) return fail(SAS_ERR_ARG, "the search kept only its top candidates (max_candidates)");
  if (r->info.peaks_only)
    return fail(SAS_ERR_ARG, "the search kept only tile-local peaks (peaks_only): its list is not complete at n_min");
  if (r->weighted) return fail(SAS_ERR_ARG, "cluster finding counts distinct epochs; this search is weighted");
  if (flags & ~SAS_PEEL_SEQUENTIAL) return fail(SAS_ERR_ARG, "unknown flags 0x%x", flags);
  if (max_clusters == 0) max_clusters = 1000;
  cudaStream_t s = (cudaStream_t)stream;
  PeelOut po;
  if (int rc = peel_clusters(result_view(r), n_min, max_clusters, (flags & SAS_PEEL_SEQUENTIAL) != 0, s, &po))
    return rc;
  sas_result* res = new sas_result();
  std::memset(res, 0, sizeof(*res));
  res->device = r->device;
  res->d_cands = po.cands;
  res->d_ids = po.ids;
  res->info = r->info;
  res->info.n_candidates = po.n;
  res->info.n_ids = po.n_ids;
  res->g = r->g;
  res->cg = r->cg;
  res->n_det = r->n_det;
  res->n_min = n_min;
  res->complete = 0;
  *out = res;
  return SAS_OK;
}

struct sas_tracks {
  int device;
  sas_track* d_tracks;
  uint32_t* d_ids;
  uint64_t n, n_ids;
};

int sas_refine(const sas_result* search, const sas_result* clusters, const sas_refine_opts* opts, void* stream,
               sas_tracks** out) {
  if (!search || !clusters || !out) return fail(SAS_ERR_ARG, "null argument");
  const bool empty = clusters->info.n_candidates == 0;
  if ((!search->d_dets || !search->d_dt) && !(empty && search->complete))
    return fail(SAS_ERR_ARG, "`search` must be a search result");
  if (clusters->n_det != search->n_det)
    return fail(SAS_ERR_ARG, "clusters come from a catalog of %llu detections, the search has %llu",
                (unsigned long long)clusters->n_det, (unsigned long long)search->n_det);
  sas_refine_opts o = opts ? *opts : sas_refine_opts{};
  if (o.n_starts == 0) o.n_starts = 500;
  if (o.n_best == 0) o.n_best = 10;
  if (o.max_csteps == 0) o.max_csteps = 100;
  if (o.max_iter == 0) o.max_iter = 10;
  if (o.radius == 0) o.radius = search->g.bin;
  if (o.n_starts > 4096) return fail(SAS_ERR_ARG, "n_starts %u above 4096", o.n_starts);
  if (o.radius < 0 || o.radius > (1 << 26)) return fail(SAS_ERR_ARG, "radius %d outside [0, 2^26]", o.radius);
  o.n_best = std::min(o.n_best, o.n_starts);
  RefineIn in;
  in.search.dets = search->d_dets;
  in.search.boff = search->d_boff;
  in.search.dt = search->d_dt;
  in.search.g = search->g;
  in.search.cg = search->cg;
  in.search.n_det = search->n_det;
  in.clusters.cands = clusters->d_cands;
  in.clusters.n = clusters->info.n_candidates;
  in.clusters.ids = clusters->d_ids;
  RefineOut ro;
  if (!empty)
    if (int rc = refine_tracks(in, o, (cudaStream_t)stream, &ro)) return rc;
  sas_tracks* t = new sas_tracks();
  t->device = search->device;
  t->d_tracks = ro.tracks;
  t->d_ids = ro.ids;
  t->n = ro.n;
  t->n_ids = ro.n_ids;
  *out = t;
  return SAS_OK;
}

int sas_tracks_get(const sas_tracks* t, sas_track* out, uint64_t cap, uint64_t* n_total, uint32_t* ids,
                   uint64_t ids_cap, uint64_t* n_ids_total, int on_device) {
  if (!t) return fail(SAS_ERR_ARG, "null tracks");
  if (n_total) *n_total = t->n;
  if (n_ids_total) *n_ids_total = t->n_ids;
  const uint64_t c1 = std::min(cap, t->n), i1 = std::min(ids_cap, t->n_ids);
  const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  if (c1) {
    if (!out) return fail(SAS_ERR_ARG, "null track buffer");
    cudaError_t e = cudaMemcpy(out, t->d_tracks, c1 * sizeof(sas_track), kind);
    if (e != cudaSuccess) return cuda_fail(e, "copy tracks");
  }
  if (i1) {
    if (!ids) return fail(SAS_ERR_ARG, "null id buffer");
    cudaError_t e = cudaMemcpy(ids, t->d_ids, i1 * sizeof(uint32_t), kind);
    if (e != cudaSuccess) return cuda_fail(e, "copy ids");
  }
  if (cap < t->n || ids_cap < t->n_ids)
    return fail(SAS_ERR_OVERFLOW, "buffers too small: need %llu tracks and %llu ids", (unsigned long long)t->n,
                (unsigned long long)t->n_ids);
  return SAS_OK;
}

void sas_tracks_free(sas_tracks* t) {
  if (!t) return;
  if (t->d_tracks) cudaFree(t->d_tracks);
  if (t->d_ids) cudaFree(t->d_ids);
  delete t;
}

int sas_owned(const sas_result* r, uint32_t n_keep, uint32_t* idx, uint64_t* n_kept, void* stream) {
  if (!r || !n_kept) return fail(SAS_ERR_ARG, "null argument");
  if (r->info.n_candidates && !idx) return fail(SAS_ERR_ARG, "null index buffer");
  return select_owned(result_view(r), n_keep, idx, n_kept, (cudaStream_t)stream);
}

int sas_peaks(const sas_result* r, uint32_t* idx, uint64_t* n_peaks, void* stream) {
  if (!r || !n_peaks) return fail(SAS_ERR_ARG, "null argument");
  if (r->info.n_candidates && !idx) return fail(SAS_ERR_ARG, "null index buffer");
  return select_peaks(result_view(r), idx, n_peaks, (cudaStream_t)stream);
}

void sas_result_free(sas_result* r) {
  if (!r) return;
  if (r->d_mem) cudaFree(r->d_mem);
  if (r->d_out) {
    cudaFree(r->d_out);
  } else {  // a cluster list: two arrays of its own
    if (r->d_cands) cudaFree(r->d_cands);
    if (r->d_ids) cudaFree(r->d_ids);
  }
  delete r;
}

int sas_cell_counts_noalloc(const sas_grid* grid, const sas_catalog* cat, const uint32_t* cells,
                            uint64_t n_cells, uint32_t* distinct, uint32_t* raw, void* stream) {
  if (!grid || !cat) return fail(SAS_ERR_ARG, "null argument");
  std::string err;
  const int rc = noalloc_cell_counts(grid->d, cat, cells, n_cells, distinct, raw, stream, &err);
  if (rc != SAS_OK) return fail(rc, "%s", err.c_str());
  return SAS_OK;
}

int sas_probe_shared_atomic_peak(uint32_t iters, void* stream, double* ops_per_s, double* sm_mhz) {
  if (!ops_per_s || !sm_mhz || iters == 0) return fail(SAS_ERR_ARG, "bad argument");
  cudaError_t e = run_atomic_probe(iters, (cudaStream_t)stream, ops_per_s, sm_mhz);
  if (e != cudaSuccess) return cuda_fail(e, "atomic probe");
  return SAS_OK;
}

int sas_probe_shared_or64_peak(uint32_t iters, void* stream, double* ops_per_s, double* sm_mhz) {
  if (!ops_per_s || !sm_mhz || iters == 0) return fail(SAS_ERR_ARG, "bad argument");
  cudaError_t e = run_or64_probe(iters, (cudaStream_t)stream, ops_per_s, sm_mhz);
  if (e != cudaSuccess) return cuda_fail(e, "64-bit atomicOr probe");
  return SAS_OK;
}

int sas_probe_shared_reduction_peak(uint32_t iters, void* stream, double* ops_per_s, double* sm_mhz) {
  if (!ops_per_s || !sm_mhz || iters == 0) return fail(SAS_ERR_ARG, "bad argument");
  cudaError_t e = run_red_probe(iters, (cudaStream_t)stream, ops_per_s, sm_mhz);
  if (e != cudaSuccess) return cuda_fail(e, "reduction probe");
  return SAS_OK;
}

}  // extern "C"
