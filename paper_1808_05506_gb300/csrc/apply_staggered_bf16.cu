// Staggered sweep, BF16 storage (kernel templates in apply_staggered_impl.cuh).
#include "apply_staggered_impl.cuh"

namespace dirac {
cudaError_t staggered_go_bf16(bool dag, const ApplyArgs& a, LaunchCfg c, cudaStream_t st) { return staggered_go_T<__nv_bfloat16>(dag, a, c, st); }
}  // namespace dirac
