// gf_inst_dir.cu -- the direction-per-warp half-sweep of small lattices (FP32-12, FP32-18, FP64-18).
#include "gf_sweep_dir.cuh"

namespace gf {

void launch_sweep_dir(int storage, int nd, const SweepArgs& a, int n_tiles, cudaStream_t s) {
#define GF_CALL(S)                                                                             \
  launch_dep(a.dep != 0,                                                                       \
             a.form == GF_OR_FIRST_ORDER                                                       \
                 ? (nd == 4 ? k_or_sweep_dir<S, 4, GF_OR_FIRST_ORDER> : k_or_sweep_dir<S, 3, GF_OR_FIRST_ORDER>) \
                 : (nd == 4 ? k_or_sweep_dir<S, 4, GF_OR_EXACT> : k_or_sweep_dir<S, 3, GF_OR_EXACT>),            \
             dim3(n_tiles), dim3(kDirThreads), 0, s, a)
  if (storage == GF_FP64_18) GF_CALL(GF_FP64_18);
  else if (storage == GF_FP32_18) GF_CALL(GF_FP32_18);
  else GF_CALL(GF_FP32_12);
#undef GF_CALL
}

}  // namespace gf
