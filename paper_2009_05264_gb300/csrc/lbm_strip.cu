// Kernel instantiations of the FP32 strip step.
#include "lbm_strip.cuh"

namespace pplbm {

cudaError_t launch_strip(int thermal, int cols, int flags, const Inst* d_inst, const Tile* d_tiles, int ntiles,
                         cudaStream_t s, const Inst* h_inst) {
  if (ntiles <= 0) return cudaSuccess;
  return thermal ? launch_strip_t<true>(cols, flags, d_inst, d_tiles, ntiles, s, h_inst)
                 : launch_strip_t<false>(cols, flags, d_inst, d_tiles, ntiles, s, h_inst);
}

cudaError_t launch_strip_persistent(int thermal, int cols, int flags, const Inst* d_inst, const Tile* d_tiles,
                                    int ntiles, int nsteps, GridBar* bar, unsigned max_polls, cudaStream_t s,
                                    const Inst* h_inst, const FlowPlan& flow) {
  if (ntiles <= 0 || nsteps <= 0) return cudaSuccess;
  return thermal ? launch_strip_persistent_t<true>(cols, flags, d_inst, d_tiles, ntiles, nsteps, bar, max_polls, s,
                                                   h_inst, flow)
                 : launch_strip_persistent_t<false>(cols, flags, d_inst, d_tiles, ntiles, nsteps, bar, max_polls, s,
                                                    h_inst, flow);
}

int strip_resident_ctas(int thermal, int cols, int flags, bool single, bool persistent) {
  return thermal ? strip_resident_t<true>(cols, flags, single, persistent)
                 : strip_resident_t<false>(cols, flags, single, persistent);
}

}  // namespace pplbm
