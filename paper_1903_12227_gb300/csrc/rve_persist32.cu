// rve_persist32.cu -- the persistent kernel on FP32 pairs (the mixed path).
#include "rve_persist.cuh"

namespace rve {

template rve_status persistent_prepare_t<float2, 0>(Plan&);
template rve_status persistent_prepare_t<float2, 1>(Plan&);
template rve_status persistent_launch<float2, 0>(const Plan&, const Ctx&, const rve_solve_opts&, cudaStream_t);
template rve_status persistent_launch<float2, 1>(const Plan&, const Ctx&, const rve_solve_opts&, cudaStream_t);

}  // namespace rve
