// Host entry to the planner of the two-level search for tests: no device work.
#include <vector>

#include "../../paper_2509_26279_gb300/csrc/sas_internal.cuh"

using namespace sas;

// Plans a search of n detections in E epochs evenly spread over `span` ticks on a
// GPU of 152 SMs.  Returns 0 (one level), 1 (two levels) or -1 (no plan).
// out: gx, gy, win, cell, units of level 1, rows of a unit, spatial tiles, list entries, counter bits, step x of the groups
extern "C" int plan_windows_for_test(const sas_grid_desc* d, uint64_t n, uint32_t E, int64_t span, int64_t tph,
                                     uint32_t n_min, double mean_weight, int64_t* out) {
  DevInfo di;
  di.sms = 152;
  di.smem_optin = 227 * 1024;
  di.smem_per_sm = 228 * 1024;
  di.ready = true;
  std::vector<int64_t> t(E);
  for (uint32_t e = 0; e < E; ++e) t[e] = E > 1 ? span * (int64_t)e / (int64_t)(E - 1) : 0;
  const uint64_t nv = (uint64_t)d->nvx * d->nvy;
  sas_opts o{};
  FieldPlan fp;
  if (plan_field(*d, n, E, t.data(), tph, n_min, 0, nv, o, di, &fp)) return -1;
  WindowPlan wp;
  if (!plan_windows(*d, n, n_min, mean_weight, 0, nv, di, fp, &wp)) return 0;
  StackArgs sa{};
  fill_window_args(wp, n_min, 0, d->nvy - 1, &sa);
  const int64_t v[] = {wp.gx, wp.gy, wp.win, wp.g.bin, (int64_t)sa.n_tiles, wp.tc.rows, (int64_t)sa.nst_x * sa.nst_y,
                       wp.list_cap, wp.tc.cb, wp.g.dvx};
  for (int i = 0; i < 10; ++i) out[i] = v[i];
  return 1;
}
