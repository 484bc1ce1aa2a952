// rve_pipe32.cu -- the fused kernels on FP32 pairs (the mixed path).
#include "rve_fused.cuh"

namespace rve {

template cudaError_t fused_step<float2, 0>(const Plan&, const Ctx&, cudaStream_t, cudaEvent_t*);
template cudaError_t fused_step<float2, 1>(const Plan&, const Ctx&, cudaStream_t, cudaEvent_t*);
template cudaError_t set_smem_attrs<float2, 0>(const Plan&);
template cudaError_t set_smem_attrs<float2, 1>(const Plan&);
template cudaError_t precond_passes<float2>(const Plan&, void*, double, const float2*, float2*, float2*, int,
                                            int, cudaStream_t);

}  // namespace rve
