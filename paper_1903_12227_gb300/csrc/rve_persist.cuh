// rve_persist.cuh -- the persistent kernel: a whole solve in one cooperative
// launch (included by the unit of each vector type).
#pragma once

#include "rve_pipeline.cuh"

namespace rve {

// ------------------------------------------------------ persistent path --
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Grid-wide barrier of a cooperative launch.  Every wait is bounded by
// timeout_ns: a block that waits longer sets the error word and leaves; all
// blocks then see the error after their own (bounded) wait and return
// false, so the kernel always ends.
inline __device__ bool grid_sync(int* ctl, unsigned nblocks, unsigned long long timeout_ns) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile int* vgen = ctl + CTL_GEN;
        volatile int* verr = ctl + CTL_ERR;
        const int gen = *vgen;
        __threadfence();
        const unsigned arrived = atomicAdd(reinterpret_cast<unsigned*>(ctl + CTL_ARRIVE), 1u);
        if (arrived == nblocks - 1) {
            atomicExch(ctl + CTL_ARRIVE, 0);
            __threadfence();
            atomicAdd(ctl + CTL_GEN, 1);
        } else {
            const unsigned long long t0 = global_ns();
            while (*vgen == gen) {
                if (*verr) break;
                if (global_ns() - t0 > timeout_ns) {
                    atomicExch(ctl + CTL_ERR, 1);
                    break;
                }
                __nanosleep(100);
            }
        }
        __threadfence();
        ok = (*verr == 0);
    }
    __syncthreads();
    return ok != 0;
}

// Control step of realization b by one warp.
inline __device__ void persist_control(const Ctx& c, int b) {
    if (c.st[b].phase == PH_DONE) return;
    const int tu0 = c.startU[b], tun = c.startU[b + 1] - tu0;
    const int tc0 = c.startC[b], tcn = c.startC[b + 1] - tc0;
    double pU[2], pC[2];
    for (int k = 0; k < 2; ++k) {
        pU[k] = warp_sum_array(c.partU + 2 * (int64_t)tu0 + k, tun, 2);
        pC[k] = warp_sum_array(c.partC + 2 * (int64_t)tc0 + k, tcn, 2);
    }
    const bool odd = threadIdx.x & 1;
    control_apply(c, b, odd ? pU[1] : pU[0], odd ? pC[1] : pC[0]);
}

struct PersistArgs {
    int tilesS, tilesU, tilesC;
    long long max_steps;
    unsigned long long timeout_ns;
};

// The whole solve in one cooperative launch: each pipeline step runs the
// refine/stencil, update, column and control phases over all tiles of the
// batch (any mix of sizes), separated by grid barriers, until every
// realization is done.
// Phases as separate (not inlined) calls, so that each keeps its own register
// allocation inside the one persistent kernel.
template <typename V, int SCHEME>
__device__ __noinline__ void phase_RS(const Ctx& c, int t) {
    fused_RS_tile<V, SCHEME, false>(c, t, DO_REFINE | DO_STENCIL);
}
template <typename V>
__device__ __noinline__ void phase_U(const Ctx& c, int t) { fused_U_tile<V>(c, t); }
template <typename V>
__device__ __noinline__ void phase_C(const Ctx& c, int t) { fused_C_tile<V>(c, c.startC, t); }

template <typename V, int SCHEME>
__global__ void __launch_bounds__(256, 2) k_persistent(const Ctx c, const PersistArgs a) {
    const unsigned nb = gridDim.x;
    for (long long step = 0; step < a.max_steps; ++step) {
        for (int t = blockIdx.x; t < a.tilesS; t += nb) phase_RS<V, SCHEME>(c, t);
        if (!grid_sync(c.ndone, nb, a.timeout_ns)) return;
        for (int t = blockIdx.x; t < a.tilesU; t += nb) phase_U<V>(c, t);
        if (!grid_sync(c.ndone, nb, a.timeout_ns)) return;
        for (int t = blockIdx.x; t < a.tilesC; t += nb) phase_C<V>(c, t);
        if (!grid_sync(c.ndone, nb, a.timeout_ns)) return;
        const int warps = blockDim.x >> 5;
        for (int r = blockIdx.x * warps + (threadIdx.x >> 5); r < c.batch; r += nb * warps)
            persist_control(c, r);
        if (!grid_sync(c.ndone, nb, a.timeout_ns)) return;
        if (*reinterpret_cast<volatile int*>(c.ndone) >= c.batch) return;
    }
}

template <typename V, int SCHEME>
rve_status persistent_prepare_t(Plan& p) {
    const size_t smem = std::max(p.smemS, std::max(p.smemU, p.smemC));
    if (cudaFuncSetAttribute(k_persistent<V, SCHEME>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem) != cudaSuccess)
        return RVE_ECUDA;
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_persistent<V, SCHEME>, 256,
                                                      smem) != cudaSuccess ||
        per_sm < 1)
        return RVE_ECUDA;
    p.persist_grid = per_sm * sms;   // co-resident: one wave
    p.persist_smem = smem;
    return RVE_OK;
}

template <typename V, int SCHEME>
rve_status persistent_launch(const Plan& p, const Ctx& c, const rve_solve_opts& o,
                                    cudaStream_t s) {
    if (p.persist_grid <= 0) return RVE_ECUDA;   // prepare_persistent() first
    PersistArgs a;
    a.tilesS = p.tilesS;
    a.tilesU = p.tilesU;
    a.tilesC = p.tilesC;
    a.max_steps = 2LL * o.max_iter + 64;
    a.timeout_ns = (unsigned long long)o.timeout_us * 1000ull;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.persist_grid);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = p.persist_smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_persistent<V, SCHEME>, c, a);
    note_launch();
    return e == cudaSuccess ? RVE_OK : RVE_ECUDA;
}

}  // namespace rve
