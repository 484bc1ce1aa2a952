// rve_pipe64.cu -- the fused kernels on double pairs (the FP64 path).
#include "rve_fused.cuh"

namespace rve {

template cudaError_t fused_step<double2, 0>(const Plan&, const Ctx&, cudaStream_t, cudaEvent_t*);
template cudaError_t fused_step<double2, 1>(const Plan&, const Ctx&, cudaStream_t, cudaEvent_t*);
template cudaError_t set_smem_attrs<double2, 0>(const Plan&);
template cudaError_t set_smem_attrs<double2, 1>(const Plan&);
template cudaError_t precond_passes<double2>(const Plan&, void*, double, const double2*, double2*, double2*, int,
                                            int, cudaStream_t);

}  // namespace rve
