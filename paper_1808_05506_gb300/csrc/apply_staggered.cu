// Dispatch of the staggered sweep on the storage type.
#include "dirac_internal.h"

namespace dirac {

cudaError_t staggered_go_f64(bool dag, const ApplyArgs& a, LaunchCfg c, cudaStream_t st);
cudaError_t staggered_go_f32(bool dag, const ApplyArgs& a, LaunchCfg c, cudaStream_t st);
cudaError_t staggered_go_bf16(bool dag, const ApplyArgs& a, LaunchCfg c, cudaStream_t st);
cudaError_t staggered_go_f16(bool dag, const ApplyArgs& a, LaunchCfg c, cudaStream_t st);

cudaError_t launch_apply_staggered(int prec, bool dag, const ApplyArgs& a, LaunchCfg c, cudaStream_t st)
{
    switch (prec) {
    case P_F64: return staggered_go_f64(dag, a, c, st);
    case P_F32: return staggered_go_f32(dag, a, c, st);
    case P_BF16: return staggered_go_bf16(dag, a, c, st);
    case P_F16: return staggered_go_f16(dag, a, c, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace dirac
