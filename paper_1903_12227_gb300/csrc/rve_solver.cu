// rve_solver.cu -- host side of the preconditioned CG for the two corrector
// problems (Sec. 3.4 and 4.1): tables, set-up and wrap-up kernels, the step
// loops and the profiler.  The pipeline's device code is in rve_pipeline.cuh.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <mutex>
#include <type_traits>
#include <vector>

#include "rve_pipeline.cuh"

namespace rve {

// ------------------------------------------------------------- tables --
// tw64[n + m] = exp(-2 pi i m / n), lap[n + m] = 4 sin^2(pi m / n) for every
// n = 2^p <= 2^maxlog, computed with sincospi/sinpi; rho[n + m] the column
// filter root for lambda = lap[n + m] and delta = 0 (1 for the singular
// column m = 0).
__global__ void k_tables(Tables out, int total) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx < 2 || idx >= total) return;
    const int p = 31 - __clz(idx);
    const int n = 1 << p, m = idx - n;
    double sn, cs;
    sincospi(-2.0 * (double)m / (double)n, &sn, &cs);
    const_cast<double2*>(out.tw64)[idx] = make_double2(cs, sn);
    const_cast<float2*>(out.tw32)[idx] = make_float2((float)cs, (float)sn);
    const_cast<int4*>(out.fx8)[idx] = fx_twiddle(cs, sn, 3);
    const_cast<int4*>(out.fx4)[idx] = fx_twiddle(cs, sn, 2);
    const double s1 = sinpi((double)m / (double)n);
    const double lam = 4.0 * s1 * s1;
    const_cast<double*>(out.lap)[idx] = lam;
    const_cast<float*>(out.lap32)[idx] = (float)lam;
    const double rho = (m == 0) ? 1.0 : filter_root(lam);
    const_cast<double*>(out.rho64)[idx] = rho;
    const_cast<float*>(out.rho32)[idx] = (float)rho;
}

Tables tables_of(const Plan& p, const void* ws) {
    const char* w = static_cast<const char*>(ws);
    Tables tb;
    tb.tw64 = reinterpret_cast<const double2*>(w + p.o_tw64);
    tb.tw32 = reinterpret_cast<const float2*>(w + p.o_tw32);
    tb.lap = reinterpret_cast<const double*>(w + p.o_lap);
    tb.lap32 = reinterpret_cast<const float*>(w + p.o_lap32);
    tb.rho64 = reinterpret_cast<const double*>(w + p.o_rho64);
    tb.rho32 = reinterpret_cast<const float*>(w + p.o_rho32);
    tb.fx8 = reinterpret_cast<const int4*>(w + p.o_fx8);
    tb.fx4 = reinterpret_cast<const int4*>(w + p.o_fx4);
    return tb;
}

cudaError_t fill_tables(const Tables& tb, int max_log2n, cudaStream_t s) {
    const int total = 2 << max_log2n;
    k_tables<<<(total + 255) / 256, 256, 0, s>>>(tb, total);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_tables(const Plan& p, void* ws, cudaStream_t s) {
    return fill_tables(tables_of(p, ws), p.max_log2n, s);
}

// One block per realization, a warp per sum (in tile order: deterministic).
// As one warp for all sums, of which the two over the stencil tiles are now
// left to finish_S, a step took 9 us at one tile and 36 us at 512.
__global__ void __launch_bounds__(128) k_control(const Ctx c) {
    __shared__ double sums[4];
    const int b = blockIdx.x;
    if (c.st[b].phase == PH_DONE) return;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t* start = w < 2 ? c.startU : c.startC;
    const double* part = (w < 2 ? c.partU : c.partC) + 2 * (int64_t)start[b] + (w & 1);
    const double v = warp_sum_array(part, start[b + 1] - start[b], 2);
    if (lane == 0) sums[w] = v;
    __syncthreads();
    if (w == 0) control_apply(c, b, sums[lane & 1], sums[2 + (lane & 1)]);
}
cudaError_t launch_control(const Plan& p, const Ctx& c, cudaStream_t s) {
    k_control<<<p.batch, 128, 0, s>>>(c);
    return cudaGetLastError();
}

__global__ void k_init(const Ctx c, int64_t nodes, size_t vbytes) {
    const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = gid; k < nodes; k += stride) {
        c.u[k] = make_double2(0.0, 0.0);
        if (vbytes == 16) {
            static_cast<double2*>(c.X)[k] = make_double2(0.0, 0.0);
            static_cast<double2*>(c.P0)[k] = make_double2(0.0, 0.0);
            static_cast<double2*>(c.P1)[k] = make_double2(0.0, 0.0);
        } else {
            static_cast<float2*>(c.X)[k] = make_float2(0.f, 0.f);
            static_cast<float2*>(c.P0)[k] = make_float2(0.f, 0.f);
            static_cast<float2*>(c.P1)[k] = make_float2(0.f, 0.f);
        }
    }
    for (int64_t b = gid; b < c.batch; b += stride) {
        RState z = {};
        z.phase = PH_REFINE;
        z.status = RVE_OK;
        c.st[b] = z;
        c.tiles_done[b] = 0;
    }
    if (gid == 0) {
        c.ndone[0] = 0;                          // realizations done
        c.ndone[CTL_ARRIVE] = 0;                 // grid barrier arrivals
        c.ndone[CTL_GEN] = 0;                    // grid barrier generation
        c.ndone[CTL_ERR] = 0;                    // a bounded wait gave up
        c.ndone[CTL_GROUPS] = 0;                 // loop groups of a captured plan
    }
}

__global__ void k_report(const Ctx c, rve_solve_info* info) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= c.batch) return;
    const RState s = c.st[b];
    rve_solve_info r;
    r.iters[0] = s.iters[0];
    r.iters[1] = s.iters[1];
    r.status = (s.phase == PH_DONE) ? s.status
               : (c.ndone[CTL_ERR] ? RVE_ETIMEOUT : RVE_ENOCONV);
    r.refinements = s.refinements;
    r.steps = s.steps;
    r.reserved = 0;
    r.relres[0] = s.relres[0];
    r.relres[1] = s.relres[1];
    info[b] = r;
}

// (double)f from the IEEE fields of a normal float or a zero, with integer
// instructions (the conversion instruction runs on the narrow FP64 pipe);
// subnormals, infinities and NaNs take the conversion instruction.
__device__ __forceinline__ double f2d(float f) {
    const unsigned b = __float_as_uint(f);
    const unsigned e = (b >> 23) & 0xFFu;
    const unsigned long long sgn = (unsigned long long)(b >> 31) << 63;
    if ((b & 0x7FFFFFFFu) == 0u) return __longlong_as_double((long long)sgn);
    if (e == 0u || e == 0xFFu) return (double)f;
    return __longlong_as_double((long long)(sgn | ((unsigned long long)(e + 896u) << 52) |
                                            ((unsigned long long)(b & 0x7FFFFFu) << 29)));
}

// Mixed path: the double-word iterate (float4 per node) becomes the caller's
// FP64 solution, in place (each thread rewrites the 16 bytes it read):
// hi + lo rounded once to double (one FP64 addition per component).
__global__ void k_u_finalize(double2* u, int64_t nodes) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nodes; k += stride) {
        const float4 w = reinterpret_cast<const float4*>(u)[k];
        u[k] = make_double2(f2d(w.x) + f2d(w.z), f2d(w.y) + f2d(w.w));
    }
}

static cudaError_t finalize_u(const Plan& p, const Ctx& c, cudaStream_t s) {
    if (p.precision != RVE_MIXED) return cudaSuccess;
    k_u_finalize<<<std::min<int64_t>((p.nodes + 255) / 256, 8 * 152), 256, 0, s>>>(c.u, p.nodes);
    note_launch();
    return cudaGetLastError();
}

// --------------------------------------------------------------- host --
std::atomic<long long> g_launches{0};

// Per-kernel event timing of the fused pipeline (diagnostics).
// Kernels: 0 refine, 1 stencil, 2 update + row transform, 3 column, 4 control.
struct Profiler {
    static constexpr int K = PROFILE_KERNELS;
    bool on = false;
    double ms[K] = {};
    long long launches[K] = {};
    std::vector<cudaEvent_t> ev;    // K + 1 events per recorded step
    int used = 0;                   // steps recorded since the last harvest
    void ensure(int steps) {
        while ((int)ev.size() < (K + 1) * steps) {
            cudaEvent_t e;
            if (cudaEventCreate(&e) != cudaSuccess) return;
            ev.push_back(e);
        }
    }
    void harvest() {   // stream already synchronised
        for (int k = 0; k < used; ++k)
            for (int j = 0; j < K; ++j) {
                float t = 0.f;
                if (cudaEventElapsedTime(&t, ev[(K + 1) * k + j], ev[(K + 1) * k + j + 1]) ==
                    cudaSuccess) {
                    ms[j] += t;
                    launches[j] += 1;
                }
            }
        used = 0;
    }
};
static Profiler g_prof;

void profile_enable(bool on) { g_prof.on = on; }
bool profile_on() { return g_prof.on; }
int profile_read(double* ms, long long* launches) {
    for (int j = 0; j < Profiler::K; ++j) {
        if (ms) ms[j] = g_prof.ms[j];
        if (launches) launches[j] = g_prof.launches[j];
        g_prof.ms[j] = 0.0;
        g_prof.launches[j] = 0;
    }
    return Profiler::K;
}

static Ctx make_ctx(const Plan& p, void* ws, const uint32_t* mask, const double* coef, double* u,
                    const rve_solve_opts& o, const double* f = nullptr) {
    char* w = static_cast<char*>(ws);
    Ctx c;
    c.batch = p.batch;
    c.desc = reinterpret_cast<const RDesc*>(w + p.o_desc);
    c.startS = reinterpret_cast<const int32_t*>(w + p.o_startS);
    c.startU = reinterpret_cast<const int32_t*>(w + p.o_startU);
    c.startC = reinterpret_cast<const int32_t*>(w + p.o_startC);
    c.st = reinterpret_cast<RState*>(w + p.o_state);
    c.partS = reinterpret_cast<double*>(w + p.o_partS);
    c.partU = reinterpret_cast<double*>(w + p.o_partU);
    c.partC = reinterpret_cast<double*>(w + p.o_partC);
    c.uscal = reinterpret_cast<double*>(w + p.o_uscal);
    c.tiles_done = reinterpret_cast<int*>(w + p.o_cnt);
    c.tb = tables_of(p, ws);
    c.cs.mask = mask;
    c.cs.coef = coef;
    c.cs.f = reinterpret_cast<const double2*>(f);
    c.u = reinterpret_cast<double2*>(u);
    c.X = w + p.o_X;
    c.R = w + p.o_R;
    c.Q = w + p.o_Q;
    c.T = w + p.o_T;
    c.P0 = w + p.o_P0;
    c.P1 = w + p.o_P1;
    c.tol = o.tol;
    c.inner_tol = (p.precision == RVE_MIXED) ? o.inner_tol : 0.5 * o.tol;
    c.delta = o.delta;
    c.max_iter = o.max_iter;
    c.ndone = reinterpret_cast<int*>(w + p.o_ctl);
    return c;
}

rve_status upload_plan(const Plan& p, void* ws, cudaStream_t s) {
    char* w = static_cast<char*>(ws);
    cudaError_t e = cudaMemcpyAsync(w + p.o_desc, p.desc.data(), sizeof(RDesc) * p.batch,
                                    cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(w + p.o_startS, p.startS.data(), sizeof(int32_t) * (p.batch + 1),
                            cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(w + p.o_startU, p.startU.data(), sizeof(int32_t) * (p.batch + 1),
                            cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(w + p.o_startC, p.startC.data(), sizeof(int32_t) * (p.batch + 1),
                            cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(w + p.o_startA, p.startA.data(), sizeof(int32_t) * (p.batch + 1),
                            cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(w + p.o_startA2, p.startA2.data(), sizeof(int32_t) * (p.batch + 1),
                            cudaMemcpyHostToDevice, s);
    for (size_t k = 0; p.cols.size() > 1 && k < p.cols.size() && e == cudaSuccess; ++k)
        e = cudaMemcpyAsync(w + p.cols[k].o_start, p.cols[k].start.data(),
                            sizeof(int32_t) * (p.batch + 1), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return RVE_ECUDA;
    return launch_tables(p, ws, s) == cudaSuccess ? RVE_OK : RVE_ECUDA;
}

template <typename V, int SCHEME>
static rve_status fused_loop(const Plan& p, const Ctx& c, const rve_solve_opts& o,
                             cudaStream_t s) {
    if (set_smem_attrs<V, SCHEME>(p) != cudaSuccess) return RVE_ECUDA;
    // bound on pipeline steps: every cycle costs one REFINE step
    const int64_t max_steps = 2LL * o.max_iter + 64;
    const int every = o.check_every > 0 ? o.check_every : 8;
    int host_done = 0;
    if (g_prof.on) {
        g_prof.ensure(every);
        g_prof.used = 0;
    }
    for (int64_t g = 0; g < max_steps; ++g) {
        cudaEvent_t* ev = nullptr;
        if (g_prof.on && (int)g_prof.ev.size() >= (Profiler::K + 1) * every)
            ev = &g_prof.ev[(Profiler::K + 1) * g_prof.used++];
        if (fused_step<V, SCHEME>(p, c, s, ev) != cudaSuccess) return RVE_ECUDA;
        if ((g + 1) % every == 0) {
            if (cudaMemcpyAsync(&host_done, c.ndone, sizeof(int), cudaMemcpyDeviceToHost, s) !=
                    cudaSuccess ||
                cudaStreamSynchronize(s) != cudaSuccess)
                return RVE_ECUDA;
            if (g_prof.on) g_prof.harvest();
            if (host_done >= p.batch) break;
        }
    }
    if (g_prof.on) {
        if (cudaStreamSynchronize(s) != cudaSuccess) return RVE_ECUDA;
        g_prof.harvest();
    }
    return RVE_OK;
}

rve_status prepare_persistent(Plan& p) {
    if (p.precision == RVE_MIXED)
        return (p.scheme == RVE_Q1_LUMPED) ? persistent_prepare_t<float2, 1>(p)
                                           : persistent_prepare_t<float2, 0>(p);
    return (p.scheme == RVE_Q1_LUMPED) ? persistent_prepare_t<double2, 1>(p)
                                       : persistent_prepare_t<double2, 0>(p);
}

// Persistent path: descriptors must already be in the workspace (upload_plan);
// everything after that is stream-ordered kernel launches (no host sync), so
// the sequence can be captured in a CUDA graph.
rve_status enqueue_solve_persistent(const Plan& p, void* ws, const uint32_t* mask,
                                    const double* coef, const rve_solve_opts& o, double* u,
                                    rve_solve_info* info, cudaStream_t s, const double* f) {
    Ctx c = make_ctx(p, ws, mask, coef, u, o, f);
    if (launch_tables(p, ws, s) != cudaSuccess) return RVE_ECUDA;
    k_init<<<std::min<int64_t>((p.nodes + 255) / 256, 4096), 256, 0, s>>>(c, p.nodes, p.vbytes);
    note_launch();
    if (cudaGetLastError() != cudaSuccess) return RVE_ECUDA;
    rve_status st;
    if (p.precision == RVE_MIXED)
        st = (p.scheme == RVE_Q1_LUMPED) ? persistent_launch<float2, 1>(p, c, o, s)
                                         : persistent_launch<float2, 0>(p, c, o, s);
    else
        st = (p.scheme == RVE_Q1_LUMPED) ? persistent_launch<double2, 1>(p, c, o, s)
                                         : persistent_launch<double2, 0>(p, c, o, s);
    if (st != RVE_OK) return st;
    if (finalize_u(p, c, s) != cudaSuccess) return RVE_ECUDA;
    k_report<<<(p.batch + 127) / 128, 128, 0, s>>>(c, info);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? RVE_OK : RVE_ECUDA;
}

// Uploads only the descriptors and tile tables (host -> device copies);
// the lookup tables are filled by a kernel in the enqueued sequence.
rve_status upload_descriptors(const Plan& p, void* ws, cudaStream_t s) {
    char* w = static_cast<char*>(ws);
    cudaError_t e = cudaMemcpyAsync(w + p.o_desc, p.desc.data(), sizeof(RDesc) * p.batch,
                                    cudaMemcpyHostToDevice, s);
    const std::vector<int32_t>* tabs[5] = {&p.startS, &p.startU, &p.startC, &p.startA, &p.startA2};
    const size_t offs[5] = {p.o_startS, p.o_startU, p.o_startC, p.o_startA, p.o_startA2};
    for (int k = 0; k < 5 && e == cudaSuccess; ++k)
        e = cudaMemcpyAsync(w + offs[k], tabs[k]->data(), sizeof(int32_t) * (p.batch + 1),
                            cudaMemcpyHostToDevice, s);
    for (size_t k = 0; p.cols.size() > 1 && k < p.cols.size() && e == cudaSuccess; ++k)
        e = cudaMemcpyAsync(w + p.cols[k].o_start, p.cols[k].start.data(),
                            sizeof(int32_t) * (p.batch + 1), cudaMemcpyHostToDevice, s);
    return e == cudaSuccess ? RVE_OK : RVE_ECUDA;
}

rve_status run_solve_persistent(const Plan& p, void* ws, const uint32_t* mask, const double* coef,
                                const rve_solve_opts& o, double* u, rve_solve_info* info,
                                cudaStream_t s, const double* f) {
    Plan q = p;
    rve_status st = (q.persist_grid > 0) ? RVE_OK : prepare_persistent(q);
    if (st == RVE_OK) st = upload_descriptors(q, ws, s);
    if (st != RVE_OK) return st;
    return enqueue_solve_persistent(q, ws, mask, coef, o, u, info, s, f);
}

// ----------------------------------------------- captured loop of steps --
// A plan captured with the fused path: the pipeline steps run inside a CUDA
// graph conditional WHILE node whose body is LOOP_GROUP fused steps (the
// same kernels as the fused path) followed by a one-thread kernel that
// re-arms the node while some realization is unfinished and the step bound
// is not reached.  No host synchronisation, so the whole solve stays inside
// one graph launch; kernel boundaries separate the phases.
constexpr int LOOP_GROUP = 4;

__global__ void k_loop_cond(cudaGraphConditionalHandle h, int* ctl, int batch,
                            long long max_groups) {
    if (threadIdx.x != 0) return;
    const int g = ctl[CTL_GROUPS] + 1;
    ctl[CTL_GROUPS] = g;
    const bool more = *reinterpret_cast<volatile int*>(ctl) < batch && g < max_groups;
    cudaGraphSetConditional(h, more ? 1u : 0u);
}

template <typename V, int SCHEME>
static rve_status loop_body(const Plan& p, const Ctx& c, cudaStream_t s,
                            cudaGraphConditionalHandle h, long long max_groups) {
    for (int k = 0; k < LOOP_GROUP; ++k)
        if (fused_step<V, SCHEME>(p, c, s, nullptr) != cudaSuccess) return RVE_ECUDA;
    k_loop_cond<<<1, 32, 0, s>>>(h, c.ndone, p.batch, max_groups);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? RVE_OK : RVE_ECUDA;
}

rve_status prepare_graph_loop(const Plan& p) {
    cudaError_t e;
    if (p.precision == RVE_MIXED)
        e = (p.scheme == RVE_Q1_LUMPED) ? set_smem_attrs<float2, 1>(p) : set_smem_attrs<float2, 0>(p);
    else
        e = (p.scheme == RVE_Q1_LUMPED) ? set_smem_attrs<double2, 1>(p) : set_smem_attrs<double2, 0>(p);
    return e == cudaSuccess ? RVE_OK : RVE_ECUDA;
}

rve_status enqueue_solve_graph_loop(const Plan& p, void* ws, const uint32_t* mask,
                                    const double* coef, const rve_solve_opts& o, double* u,
                                    rve_solve_info* info, cudaStream_t s, const double* f) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaGraph_t g = nullptr;
    const cudaGraphNode_t* deps = nullptr;
    size_t nd = 0;
    if (cudaStreamGetCaptureInfo(s, &cs, nullptr, &g, &deps, nullptr, &nd) != cudaSuccess ||
        cs != cudaStreamCaptureStatusActive)
        return RVE_EINVAL;   // only inside a stream capture
    Ctx c = make_ctx(p, ws, mask, coef, u, o, f);
    if (launch_tables(p, ws, s) != cudaSuccess) return RVE_ECUDA;
    k_init<<<std::min<int64_t>((p.nodes + 255) / 256, 4096), 256, 0, s>>>(c, p.nodes, p.vbytes);
    note_launch();
    if (cudaGetLastError() != cudaSuccess) return RVE_ECUDA;
    if (cudaStreamGetCaptureInfo(s, &cs, nullptr, &g, &deps, nullptr, &nd) != cudaSuccess)
        return RVE_ECUDA;
    const std::vector<cudaGraphNode_t> dep(deps, deps + nd);   // valid until the next call
    // the conditional node, run at least once per graph launch (default 1,
    // re-assigned on every launch)
    cudaGraphConditionalHandle h;
    if (cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault) != cudaSuccess)
        return RVE_ECUDA;
    cudaGraphNodeParams np = {};
    np.type = cudaGraphNodeTypeConditional;
    np.conditional.handle = h;
    np.conditional.type = cudaGraphCondTypeWhile;
    np.conditional.size = 1;
    cudaGraphNode_t node;
    if (cudaGraphAddNode(&node, g, dep.data(), nullptr, dep.size(), &np) != cudaSuccess)
        return RVE_ECUDA;
    cudaGraph_t body = np.conditional.phGraph_out[0];
    if (cudaStreamUpdateCaptureDependencies(s, &node, nullptr, 1,
                                            cudaStreamSetCaptureDependencies) != cudaSuccess)
        return RVE_ECUDA;
    // the body: LOOP_GROUP pipeline steps and the re-arming kernel, captured
    // on a helper stream straight into the node's body graph
    cudaStream_t sb = nullptr;
    if (cudaStreamCreateWithFlags(&sb, cudaStreamNonBlocking) != cudaSuccess) return RVE_ECUDA;
    rve_status st = RVE_OK;
    if (cudaStreamBeginCaptureToGraph(sb, body, nullptr, nullptr, 0,
                                      cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
        st = RVE_ECUDA;
    } else {
        const long long max_groups = (2LL * o.max_iter + 64) / LOOP_GROUP + 1;
        if (p.precision == RVE_MIXED)
            st = (p.scheme == RVE_Q1_LUMPED) ? loop_body<float2, 1>(p, c, sb, h, max_groups)
                                             : loop_body<float2, 0>(p, c, sb, h, max_groups);
        else
            st = (p.scheme == RVE_Q1_LUMPED) ? loop_body<double2, 1>(p, c, sb, h, max_groups)
                                             : loop_body<double2, 0>(p, c, sb, h, max_groups);
        cudaGraph_t out = nullptr;
        if (cudaStreamEndCapture(sb, &out) != cudaSuccess) st = RVE_ECUDA;
    }
    cudaStreamDestroy(sb);
    if (st != RVE_OK) return st;
    if (finalize_u(p, c, s) != cudaSuccess) return RVE_ECUDA;
    k_report<<<(p.batch + 127) / 128, 128, 0, s>>>(c, info);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? RVE_OK : RVE_ECUDA;
}

rve_status run_solve_fused(const Plan& p, void* ws, const uint32_t* mask, const double* coef,
                           const rve_solve_opts& o, double* u, rve_solve_info* info,
                           cudaStream_t s, const double* f) {
    rve_status st = upload_plan(p, ws, s);
    if (st != RVE_OK) return st;
    Ctx c = make_ctx(p, ws, mask, coef, u, o, f);
    k_init<<<std::min<int64_t>((p.nodes + 255) / 256, 4096), 256, 0, s>>>(c, p.nodes, p.vbytes);
    note_launch();
    if (cudaGetLastError() != cudaSuccess) return RVE_ECUDA;
    if (p.precision == RVE_MIXED) {
        st = (p.scheme == RVE_Q1_LUMPED) ? fused_loop<float2, 1>(p, c, o, s)
                                         : fused_loop<float2, 0>(p, c, o, s);
    } else {
        st = (p.scheme == RVE_Q1_LUMPED) ? fused_loop<double2, 1>(p, c, o, s)
                                         : fused_loop<double2, 0>(p, c, o, s);
    }
    if (st != RVE_OK) return st;
    if (finalize_u(p, c, s) != cudaSuccess) return RVE_ECUDA;
    k_report<<<(p.batch + 127) / 128, 128, 0, s>>>(c, info);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? RVE_OK : RVE_ECUDA;
}

cudaError_t launch_precond(const Plan& p, void* ws, double delta, int precision, const void* x,
                           void* y, cudaStream_t s) {
    if (upload_plan(p, ws, s) != RVE_OK) return cudaErrorUnknown;
    char* w = static_cast<char*>(ws);
    if (precision == RVE_FP64)
        return precond_passes<double2>(p, ws, delta, static_cast<const double2*>(x),
                                       static_cast<double2*>(y),
                                       reinterpret_cast<double2*>(w + p.o_T), 0, p.batch, s);
    return precond_passes<float2>(p, ws, delta, static_cast<const float2*>(x),
                                  static_cast<float2*>(y), reinterpret_cast<float2*>(w + p.o_T), 0,
                                  p.batch, s);
}

}  // namespace rve
