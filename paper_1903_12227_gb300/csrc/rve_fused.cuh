// rve_fused.cuh -- kernels and launchers of the fused path and of the
// standalone preconditioner (included by the unit of each vector type).
#pragma once

#include "rve_pipeline.cuh"

namespace rve {

// One launch per pipeline kernel (the fused path).
// The refine and the stencil pass share a launch: a refining realization's
// blocks compute the true residual where the others run the stencil.  (As a
// launch of its own the refine pass had nothing to do in 9 of 10 steps and its
// blocks still took 10 us a step at 4600 blocks, 2 us at one.)
template <typename V, int SCHEME>
__global__ void __launch_bounds__(256, sizeof(V) == 8 ? 3 : 2) k_fused_RS(const Ctx c, int which) {
    fused_RS_tile<V, SCHEME, true>(c, blockIdx.x, which);
}
template <typename V, int SCHEME>
__global__ void __launch_bounds__(256, sizeof(V) == 8 ? 3 : 2) k_fused_Q(const Ctx c) {
    fused_Q_tile<V, SCHEME>(c, blockIdx.x);
}
template <typename V>
__global__ void __launch_bounds__(256, sizeof(V) == 8 ? 4 : 2) k_fused_U(const Ctx c) { fused_U_tile<V>(c, blockIdx.x); }
template <typename V>
__global__ void __launch_bounds__(512) k_fused_C(const Ctx c, const int32_t* __restrict__ start) {
    fused_C_tile<V>(c, start, blockIdx.x);
}

template <typename V, int SCHEME>
cudaError_t fused_step(const Plan& p, const Ctx& c, cudaStream_t s, cudaEvent_t* ev) {
    if (ev) {   // profiling: the two halves apart
        cudaEventRecord(ev[0], s);
        k_fused_RS<V, SCHEME><<<p.tilesS, 256, p.smemS, s>>>(c, DO_REFINE);
        cudaEventRecord(ev[1], s);
        k_fused_RS<V, SCHEME><<<p.tilesS, 256, p.smemS, s>>>(c, DO_STENCIL);
        note_launch();
    } else {
        k_fused_RS<V, SCHEME><<<p.tilesS, 256, p.smemS, s>>>(c, DO_REFINE | DO_STENCIL);
    }
    if (p.split) {
        k_fused_Q<V, SCHEME><<<p.tilesS, 256, 0, s>>>(c);
        note_launch();
    }
    if (ev) cudaEventRecord(ev[2], s);
    k_fused_U<V><<<p.tilesU, 256, p.smemU, s>>>(c);
    if (ev) cudaEventRecord(ev[3], s);
    // a launch per block width: with one width for the batch, that of its largest
    // grid, the sums of the smaller ones depended on their company.  The tail of
    // the second launch costs batches that mix widths 2 to 4 % (one 2048^2 and 60
    // 512^2 grids 30.5 -> 31.2 ms, with 300 of 64^2 13.0 -> 13.5 ms)
    const char* w = reinterpret_cast<const char*>(c.startC) - p.o_startC;
    for (const ColClass& k : p.cols)
        k_fused_C<V><<<k.tiles, k.threads, k.smem, s>>>(c, reinterpret_cast<const int32_t*>(w + k.o_start));
    if (ev) cudaEventRecord(ev[4], s);
    const cudaError_t ce = launch_control(p, c, s);
    if (ce != cudaSuccess) return ce;
    if (ev) cudaEventRecord(ev[5], s);
    note_launch(3 + (int)p.cols.size());
    return cudaGetLastError();
}

template <typename V, int SCHEME>
cudaError_t set_smem_attrs(const Plan& p) {
    cudaError_t e = cudaFuncSetAttribute(k_fused_RS<V, SCHEME>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smemS);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_fused_U<V>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)p.smemU);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_fused_C<V>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)p.smemC);
    return e;
}

// --------------------------------------------------- preconditioner apply --
// Standalone transform passes (rve_apply_precond and the plain path): row
// Hartley of `in` into `out`, and the column pair with the scale in place.
// Tiles tile0 .. tile0 + gridDim.x - 1 of the batch's row / column tiling.
template <typename V>
__global__ void __launch_bounds__(256, sizeof(V) == 8 ? 3 : 2) k_row_hartley(const RDesc* __restrict__ desc,
                                                     const int32_t* __restrict__ startU, int batch,
                                                     int tile0, Tables tb, const V* __restrict__ in,
                                                     V* __restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned fxs[8];
    const int blk = blockIdx.x + tile0;
    const int b = find_real(startU, batch, blk);
    const RDesc d = desc[b];
    dispatch_size(d.log2n, [&]<int LG>() {
        const RowLayout<LG> L(d.log2n);
        const TeamBar team(L.qq, L.z.T);
        const int row0 = (blk - startU[b]) * d.tU;
        for (int g0 = 0; g0 < d.tU; g0 += L.G) {
            const bool active = g0 + L.qq < d.tU;
            const int row = row0 + g0 + L.qq;
            V* buf = reinterpret_cast<V*>(smem_raw) + (active ? L.qq : 0) * seq_stride(L.z.n);
            V v[8];
            if (active) {
#pragma unroll
                for (int m = 0; m < 8; ++m) v[m] = in[node_at(d, L.z, row, L.t + m * L.z.T)];
            }
            hartley_row<LG>(v, buf, L.t, twiddles<V>(tb, L.z.n), fx_twiddles(tb, L.z.n), active,
                            fxs, team);
            if (active) {
#pragma unroll
                for (int m = 0; m < 8; ++m) out[node_at(d, L.z, row, L.t + m * L.z.T)] = v[m];
            }
            team();   // mirror reads of the buffers are done
        }
    });
}

template <typename V>
__global__ void __launch_bounds__(512) k_col_hartley(const RDesc* __restrict__ desc,
                                                      const int32_t* __restrict__ startC, int batch,
                                                      int tile0, Tables tb, double delta,
                                                      V* __restrict__ T) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[64];   // block_sum2 scratch: 4 floats per warp (<= 32 warps)
    const int blk = blockIdx.x + tile0;
    const int b = find_real(startC, batch, blk);
    const RDesc d = desc[b];
    col_transform_tile<V>(T, T, d, (blk - startC[b]) * d.tC, reinterpret_cast<V*>(smem_raw), tb,
                          delta, red, nullptr);
}

template <typename V>
cudaError_t precond_passes(const Plan& p, void* ws, double delta, const V* x, V* y, V* tmp,
                           int b_first, int b_count, cudaStream_t s) {
    char* w = static_cast<char*>(ws);
    const RDesc* desc = reinterpret_cast<const RDesc*>(w + p.o_desc);
    const int32_t* startU = reinterpret_cast<const int32_t*>(w + p.o_startU);
    const Tables tb = tables_of(p, ws);
    cudaError_t e = cudaFuncSetAttribute(k_row_hartley<V>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smemU);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_col_hartley<V>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)p.smemC);
    if (e != cudaSuccess) return e;
    const int u0 = p.startU[b_first], un = p.startU[b_first + b_count] - u0;
    k_row_hartley<V><<<un, 256, p.smemU, s>>>(desc, startU, p.batch, u0, tb, x, tmp);
    int launches = 2;
    for (const ColClass& k : p.cols) {
        const int c0 = k.start[b_first], cn = k.start[b_first + b_count] - c0;
        if (cn == 0) continue;
        k_col_hartley<V><<<cn, k.threads, k.smem, s>>>(desc, reinterpret_cast<const int32_t*>(w + k.o_start),
                                                       p.batch, c0, tb, delta, tmp);
        ++launches;
    }
    k_row_hartley<V><<<un, 256, p.smemU, s>>>(desc, startU, p.batch, u0, tb, tmp, y);
    note_launch(launches);
    return cudaGetLastError();
}

}  // namespace rve
