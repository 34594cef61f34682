// The stack kernel's instantiations of the window search (sas_hier.cu): tiles of
// 4 x 4 groups of lattice points, 8-bit counters for detections and 16-bit ones
// for weights and for detections whose 8-bit counters wrapped.  Four columns of groups share the row's address, and 16 points a
// tile leave room for tiles of some 100 x 100 cells, whose overlap (2 cells) and
// shift spread (about a third of a tile) stay small.
#include "sas_stack_kernel.cuh"

namespace sas {

#define SAS_WINDOW_CONFIGS(X) X(4, 4, 8) X(4, 4, 16)

cudaError_t launch_stack_windows(const StackArgs& a, int grid, cudaStream_t s) {
#define SAS_LAUNCH(KX, KY, CB) \
  if (a.tc.kx == KX && a.tc.ky == KY && a.tc.cb == CB) return launch_t<KX, KY, CB, kModeWindows>(a, grid, s);
  SAS_WINDOW_CONFIGS(SAS_LAUNCH)
#undef SAS_LAUNCH
  return cudaErrorInvalidValue;
}

cudaError_t stack_set_smem_attr_windows(int kx, int ky, int cb, size_t smem) {
#define SAS_ATTR(KX, KY, CB) \
  if (kx == KX && ky == KY && cb == CB)    \
    return raise_smem_limit((const void*)k_stack<KX, KY, CB, false, kModeWindows>, smem);
  SAS_WINDOW_CONFIGS(SAS_ATTR)
#undef SAS_ATTR
  return cudaErrorInvalidValue;
}

}  // namespace sas
