// rve_persist64.cu -- the persistent kernel on double pairs (the FP64 path).
#include "rve_persist.cuh"

namespace rve {

template rve_status persistent_prepare_t<double2, 0>(Plan&);
template rve_status persistent_prepare_t<double2, 1>(Plan&);
template rve_status persistent_launch<double2, 0>(const Plan&, const Ctx&, const rve_solve_opts&, cudaStream_t);
template rve_status persistent_launch<double2, 1>(const Plan&, const Ctx&, const rve_solve_opts&, cudaStream_t);

}  // namespace rve
