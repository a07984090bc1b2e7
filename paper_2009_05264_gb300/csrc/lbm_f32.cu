// Kernel instantiations for float storage and arithmetic.
#include "lbm_kernels.cuh"
#include "lbm_tma.cuh"

namespace pplbm {

cudaError_t launch_lbm_f32(int thermal, int cols, int mode, int kernel, bool full, const Inst* d_inst,
                          const Tile* d_tiles, int ntiles, cudaStream_t s, const Inst* h_inst, unsigned max_polls) {
  if (mode == MODE_STEP && kernel == LBM_KERNEL_TMA)
    return launch_tma(thermal, cols, d_inst, d_tiles, ntiles, s, h_inst, max_polls);
  return launch_precision<float>(thermal, cols, mode, full, false, d_inst, d_tiles, ntiles, s, h_inst);
}

cudaError_t launch_persistent_f32(int thermal, int cols, int kernel, bool full, const Inst* d_inst,
                                  const Tile* d_tiles, int ntiles, int nsteps, GridBar* bar, unsigned max_polls,
                                  cudaStream_t s, const Inst* h_inst, const FlowPlan& flow) {
  if (kernel != LBM_KERNEL_SCALAR) return cudaErrorNotSupported;
  return launch_persistent_precision<float>(thermal, cols, full, false, d_inst, d_tiles, ntiles, nsteps, bar, max_polls,
                                            s, h_inst, flow);
}

int persistent_resident_f32(int thermal, int cols, int, bool full, bool single) {
  return persistent_resident_precision<float>(thermal, cols, full, false, single);
}

int strip_resident_ctas(int thermal, int cols, int flags, bool single, bool persistent);

int resident_ctas_f32(int thermal, int cols, int kernel, int flags) {
  if (kernel == FORM_STRIP) return strip_resident_ctas(thermal, cols, flags, true, false);
  if (kernel == LBM_KERNEL_TMA && cols == ST_COLS) return resident_tma(thermal);
  return resident_precision<float>(thermal, cols, false);
}

cudaError_t launch_init_from_fields_f32(const Inst* d_inst, int nx, int ny, const double* d_fields, int has_T,
                                       cudaStream_t s) {
  return launch_init_fields_t<float>(d_inst, nx, ny, d_fields, has_T, s);
}

cudaError_t launch_init_builtin_f32(const Inst* d_inst, int nx, int ny, InitSpec spec, cudaStream_t s) {
  return launch_init_builtin_t<float>(d_inst, nx, ny, spec, s);
}

}  // namespace pplbm
