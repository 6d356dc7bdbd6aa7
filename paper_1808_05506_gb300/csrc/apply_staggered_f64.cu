// Staggered sweep, FP64 storage (kernel templates in apply_staggered_impl.cuh).
#include "apply_staggered_impl.cuh"

namespace dirac {
cudaError_t staggered_go_f64(bool dag, const ApplyArgs& a, LaunchCfg c, cudaStream_t st) { return staggered_go_T<double>(dag, a, c, st); }
}  // namespace dirac
