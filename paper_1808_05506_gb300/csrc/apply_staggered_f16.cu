// Staggered sweep, FP16 storage (kernel templates in apply_staggered_impl.cuh).
#include "apply_staggered_impl.cuh"

namespace dirac {
cudaError_t staggered_go_f16(bool dag, const ApplyArgs& a, LaunchCfg c, cudaStream_t st) { return staggered_go_T<__half>(dag, a, c, st); }
}  // namespace dirac
