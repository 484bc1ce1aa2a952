// rve_ops.cu -- field generation, right-hand sides, stiffness apply,
// homogenized matrix and its adjoint (sm_103a).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "rve_ahom.cuh"
#include "rve_common.cuh"
#include "rve_internal.h"

namespace rve {

// uniform integer below n: high word of the 128-bit product (Lemire 2019,
// no rejection)
__device__ __forceinline__ int uniform_below(uint64_t v, uint32_t n) {
    return (int)__umul64hi(v, (uint64_t)n);
}
constexpr uint32_t TAG_CORNER = 1u;

// One thread per (inclusion, row of its square): sets the square's cells of
// that row in the bitmask (Eq. "Stoch-decomp": the covered set is the union
// of the inclusions, overlaps allowed, periodic wrap).
__global__ void k_gen_field(const __grid_constant__ DescChunk ch, uint32_t* __restrict__ mask) {
    const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= ch.start[ch.count]) return;
    const int b = find_real(ch.start, ch.count, (int)gid);
    const RDesc& d = ch.d[b];
    const int w = (int)gid - ch.start[b];
    const int k = w / d.s, d1 = w - k * d.s;
    const int c1 = uniform_below(sm64_draw(d.key, TAG_CORNER, 2ull * k), (uint32_t)d.n);
    const int c2 = uniform_below(sm64_draw(d.key, TAG_CORNER, 2ull * k + 1), (uint32_t)d.n);
    const int i1 = (c1 + d1) & (d.n - 1);
    uint32_t* row = mask + d.word_off + (((int64_t)i1 * d.n) >> 5);
    // columns c2 .. c2+s-1 (mod n), split at the wrap, then into words
    int j = c2, left = d.s;
    while (left > 0) {
        const int run = min(left, d.n - j);   // until the wrap
        int jj = j, rl = run;
        while (rl > 0) {
            const int bit = jj & 31;
            const int take = min(rl, 32 - bit);
            const uint32_t m = (take == 32) ? 0xffffffffu : (((1u << take) - 1u) << bit);
            atomicOr(row + (jj >> 5), m);
            jj += take;
            rl -= take;
        }
        left -= run;
        j = 0;
    }
}

// ------------------------------------------------------ RHS / stiffness --
// Work unit = 256 nodes (n*n is a multiple of 1024 for n >= 32).
constexpr int NODE_TILE = 256;

__global__ void k_rhs(const __grid_constant__ DescChunk ch, CoefSrc cs, double2* __restrict__ f) {
    const int b = find_real(ch.start, ch.count, blockIdx.x);
    const RDesc& d = ch.d[b];
    const int64_t node = (int64_t)(blockIdx.x - ch.start[b]) * NODE_TILE + threadIdx.x;
    const int i = (int)(node >> d.log2n), j = (int)(node & (d.n - 1));
    f[d.node_off + node] = rhs_at(cells_at(cs, d, i, j), d.h);
}

// Cell values a_c from the bitmask and the two values (one thread per cell).
__global__ void k_coef_from_mask(const __grid_constant__ DescChunk ch, const uint32_t* __restrict__ mask,
                                 double* __restrict__ coef) {
    const int b = find_real(ch.start, ch.count, blockIdx.x);
    const RDesc& d = ch.d[b];
    const int64_t cell = (int64_t)(blockIdx.x - ch.start[b]) * NODE_TILE + threadIdx.x;
    const uint32_t w = __ldg(mask + d.word_off + (cell >> 5));
    coef[d.node_off + cell] = ((w >> (cell & 31)) & 1u) ? d.a_incl : d.a_matrix;
}

template <typename V>
__device__ __forceinline__ V ldv(const V* __restrict__ x, const RDesc& d, int i, int j) {
    return x[d.node_off + ((int64_t)(i & (d.n - 1)) << d.log2n) + (j & (d.n - 1))];
}

// y = A x.  A thread walks down `rows` rows of one column (FP64) or two (FP32)
// with the 3 x 3 neighbourhood in registers, so that a node costs the loads of
// its row's new neighbours; 256 threads take min(n, 256) columns (FP32: min(n,
// 512)) and, on smaller grids, several groups of rows.  FP32: the cell values
// stay in FP32 -- through double, as the cell accessor returns them, every node
// cost four conversions on the FP64 pipe -- and the kernel is bound by memory:
// 96 x 512^2 nodes 250 -> 96 us.  FP64: bound by the FP64 pipe (StencilRow);
// 11 x 1024^2 nodes, explicit cells 629 -> 566 us.
constexpr int STIFF_THREADS = 256;
template <typename V> __host__ __device__ constexpr int stiff_cols(int n) {   // columns of a block
    return n < (int)(4096 / sizeof(V)) ? n : (int)(4096 / sizeof(V));
}
// Rows of a block: `rows` per thread and group.
template <typename V> __host__ __device__ constexpr int stiff_block_rows(int n, int rows) {
    const int groups = STIFF_THREADS / (stiff_cols<V>(n) / (int)(16 / sizeof(V)));
    return groups * rows < n ? groups * rows : n;
}

template <int SCHEME, typename V>
__global__ void __launch_bounds__(STIFF_THREADS) k_stiffness(const __grid_constant__ DescChunk ch,
                                                             CoefSrc cs, const V* __restrict__ x,
                                                             V* __restrict__ y, int rows,
                                                             bool pairs) {
    __shared__ __align__(16) double rowtab[sizeof(V) == 16 ? ROW_TABLE : 2];
    const int b = find_real(ch.start, ch.count, blockIdx.x);
    const RDesc& d = ch.d[b];
    const int n = d.n, m = n - 1, lg = d.log2n;
    constexpr int CPT = 16 / sizeof(V);                     // columns of a thread
    const int CW = stiff_cols<V>(n), BR = stiff_block_rows<V>(n, rows);
    const int across = CW / CPT, groups = STIFF_THREADS / across;
    const int per = (BR + groups - 1) / groups;             // rows of a thread
    const int blk = blockIdx.x - ch.start[b], cblks = n / CW;
    const int g = threadIdx.x / across;
    const int j = (blk % cblks) * CW + CPT * (threadIdx.x - g * across);
    const int i0 = (blk / cblks) * BR + g * per, i1 = min(i0 + per, (blk / cblks) * BR + BR);
    const V* __restrict__ xb = x + d.node_off;
    V* __restrict__ yb = y + d.node_off;
    const uint32_t* __restrict__ mw = cs.coef ? nullptr : cs.mask + d.word_off;
    const double* __restrict__ cf = cs.coef ? cs.coef + d.node_off : nullptr;
    const int jm = (j - 1) & m, jp = (j + CPT) & m;
    // bits of cells (i, j - 1), (i, j), (i, j + 1) (j even for FP32, so the last two share a word)
    auto bits = [&](int i) -> unsigned {
        const int64_t r = (int64_t)(i & m) << lg;
        const uint32_t w = __ldg(mw + ((r + j) >> 5)) >> (j & 31);
        const uint32_t v = (j & 31) ? __ldg(mw + ((r + j) >> 5)) >> ((j & 31) - 1)
                                    : __ldg(mw + ((r + jm) >> 5)) >> 31;
        return (v & 1u) | ((w & 3u) << 1);
    };
    if constexpr (sizeof(V) == 16) {
        if (mw) {
            fill_row_table<SCHEME>(rowtab, d.a_matrix, d.a_incl);
            __syncthreads();
        }
        if (i0 >= i1) return;
        auto at = [&](int i, int jj) { return __ldg(xb + ((int64_t)(i & m) << lg) + jj); };
        V u0 = at(i0 - 1, jm), u1 = at(i0 - 1, j), u2 = at(i0 - 1, jp);
        V m0 = at(i0, jm), m1 = at(i0, j), m2 = at(i0, jp);
        auto row = [&](const StencilRow& w, int i, const V& d0, const V& d1, const V& d2, auto doubled) {
            constexpr double IK = 1.0 / row_scale<SCHEME>();
            V q = apply_row<SCHEME, decltype(doubled)::value>(w, u0, u1, u2, m0, m1, m2, d0, d1, d2);
            q = make_double2(IK * q.x, IK * q.y);
            // K A x overflows where A x need not: again with the weights over 8
            if (max((unsigned)__double2hiint(q.x) & 0x7FFFFFFFu, (unsigned)__double2hiint(q.y) & 0x7FFFFFFFu) >= 0x7FF00000u) {
                q = apply_row<SCHEME, decltype(doubled)::value>(over_8<SCHEME>(w), u0, u1, u2, m0, m1, m2, d0, d1, d2);
                q = make_double2(8.0 * IK * q.x, 8.0 * IK * q.y);
            }
            yb[((int64_t)i << lg) + j] = q;
            u0 = m0; u1 = m1; u2 = m2;
            m0 = d0; m1 = d1; m2 = d2;
        };
        if (mw) {
            unsigned top = bits(i0 - 1) & 3u;
#pragma unroll 2
            for (int i = i0; i < i1; ++i) {
                const V d0 = at(i + 1, jm), d1 = at(i + 1, j), d2 = at(i + 1, jp);
                const unsigned bot = bits(i) & 3u;
                row(table_row<SCHEME>(rowtab, top | (bot << 2)), i, d0, d1, d2, std::true_type());
                top = bot;
            }
        } else {
            auto cell = [&](int i, int jj) { return __ldg(cf + ((int64_t)(i & m) << lg) + jj); };
            RowWalk<SCHEME> walk(cell(i0 - 1, jm), cell(i0 - 1, j));
#pragma unroll 2
            for (int i = i0; i < i1; ++i) {
                const V d0 = at(i + 1, jm), d1 = at(i + 1, j), d2 = at(i + 1, jp);
                row(walk.step(cell(i, jm), cell(i, j)), i, d0, d1, d2, std::false_type());
            }
        }
    } else {
        if (i0 >= i1) return;
        const float ai = (float)d.a_incl, am = (float)d.a_matrix;
        struct Row { V l, a, b, r; };     // x at j - 1, j, j + 1, j + 2
        struct Cel { float l, a, b; };    // cells j - 1, j, j + 1
        // `pairs`: x and y are 16-byte aligned (the ABI asks for 8)
        auto xrow = [&](int i) -> Row {
            const V* p = xb + ((int64_t)(i & m) << lg);
            float4 c;
            if (pairs) {
                c = __ldg(reinterpret_cast<const float4*>(p + j));
            } else {
                const V a = __ldg(p + j), b2 = __ldg(p + j + 1);
                c = make_float4(a.x, a.y, b2.x, b2.y);
            }
            return Row{__ldg(p + jm), make_float2(c.x, c.y), make_float2(c.z, c.w), __ldg(p + jp)};
        };
        auto crow = [&](int i) -> Cel {
            if (mw) {
                const unsigned k = bits(i);
                return Cel{(k & 1u) ? ai : am, (k & 2u) ? ai : am, (k & 4u) ? ai : am};
            }
            const double* p = cf + ((int64_t)(i & m) << lg);
            return Cel{(float)__ldg(p + jm), (float)__ldg(p + j), (float)__ldg(p + j + 1)};
        };
        Row u = xrow(i0 - 1), c = xrow(i0), ahead = xrow(i0 + 1);   // one row ahead of its use
        Cel t = crow(i0 - 1), o = crow(i0);
#pragma unroll 4
        for (int i = i0; i < i1; ++i) {
            const Row dn = ahead;
            ahead = xrow(i + 2);
            const Cel on = crow(i + 1);
            const V q0 = stencil_apply<SCHEME, V>(CellsT<float>{t.l, t.a, o.l, o.a}, u.l, u.a, u.b, c.l, c.a,
                                                  c.b, dn.l, dn.a, dn.b);
            const V q1 = stencil_apply<SCHEME, V>(CellsT<float>{t.a, t.b, o.a, o.b}, u.a, u.b, u.r, c.a, c.b,
                                                  c.r, dn.a, dn.b, dn.r);
            V* o2 = yb + ((int64_t)i << lg) + j;
            if (pairs) {
                *reinterpret_cast<float4*>(o2) = make_float4(q0.x, q0.y, q1.x, q1.y);
            } else {
                o2[0] = q0;
                o2[1] = q1;
            }
            u = c;
            c = dn;
            t = o;
            o = on;
        }
    }
}

// y = M x, M = M1 (x) M1 the Q1 mass matrix (1D: consistent h [1/6, 2/3,
// 1/6], lumped h [0, 1, 0]), periodic 9-point (resp. 1-point) stencil: the
// load vector of a nodal load for the general-right-hand-side solve.
template <int SCHEME>
__global__ void k_mass(const __grid_constant__ DescChunk ch, const double2* __restrict__ x,
                       double2* __restrict__ y) {
    const int b = find_real(ch.start, ch.count, blockIdx.x);
    const RDesc& d = ch.d[b];
    const int64_t node = (int64_t)(blockIdx.x - ch.start[b]) * NODE_TILE + threadIdx.x;
    const int i = (int)(node >> d.log2n), j = (int)(node & (d.n - 1));
    const double h2 = d.h * d.h;
    double2 acc = make_double2(0.0, 0.0);
    if (SCHEME == 1) {
        acc = ldv(x, d, i, j);
    } else {
        const double w[3] = {1.0 / 6.0, 2.0 / 3.0, 1.0 / 6.0};
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double2 v = ldv(x, d, i + a - 1, j + c - 1);
                acc.x = fma(w[a] * w[c], v.x, acc.x);
                acc.y = fma(w[a] * w[c], v.y, acc.y);
            }
    }
    y[d.node_off + node] = make_double2(h2 * acc.x, h2 * acc.y);
}

// --------------------------------------------------- Chebyshev moments --
// One step of the Chebyshev recurrence of A~ = a0 A - a1 I for both start
// vectors of every realization (the spectral-density appendix):
//   w_{k+1} = 2 A~ w_k - w_{k-1}   (first step: w_1 = A~ w_0),
// written over w_{k-1}; per tile of NODE_TILE nodes the partial sums
// w_k.w_k and w_{k+1}.w_k per start vector, from which the moments follow by
// T_2k = 2 T_k^2 - T_0 and T_{2k+1} = 2 T_{k+1} T_k - T_1 (two moments per
// operator application).  FP64 throughout.
template <int SCHEME>
__global__ void __launch_bounds__(NODE_TILE) k_cheb(const __grid_constant__ DescChunk ch,
                                                    CoefSrc cs, double a0, double a1, int first,
                                                    const double2* __restrict__ wc,
                                                    double2* __restrict__ wp,
                                                    double* __restrict__ part) {
    __shared__ double red[8];
    const int b = find_real(ch.start, ch.count, blockIdx.x);
    const RDesc& d = ch.d[b];
    const int64_t node = (int64_t)(blockIdx.x - ch.start[b]) * NODE_TILE + threadIdx.x;
    const int i = (int)(node >> d.log2n), j = (int)(node & (d.n - 1));
    const Cells4 a = cells_at(cs, d, i, j);
    const double2 Aw = stencil_apply<SCHEME, double2>(
        a, ldv(wc, d, i - 1, j - 1), ldv(wc, d, i - 1, j), ldv(wc, d, i - 1, j + 1),
        ldv(wc, d, i, j - 1), ldv(wc, d, i, j), ldv(wc, d, i, j + 1),
        ldv(wc, d, i + 1, j - 1), ldv(wc, d, i + 1, j), ldv(wc, d, i + 1, j + 1));
    const double2 w = wc[d.node_off + node];
    double2 t = make_double2(a0 * Aw.x - a1 * w.x, a0 * Aw.y - a1 * w.y);
    if (!first) {
        const double2 wm = wp[d.node_off + node];
        t = make_double2(2.0 * t.x - wm.x, 2.0 * t.y - wm.y);
    }
    wp[d.node_off + node] = t;
    const double v[4] = {w.x * w.x, w.y * w.y, t.x * w.x, t.y * w.y};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const double sum = block_sum(v[k], red);
        if (threadIdx.x == 0) part[(int64_t)blockIdx.x * 4 + k] = sum;
    }
}

// The whole recurrence of a realization of n <= 128 in one cluster of eight
// blocks: block r keeps its n / 8 rows of w_k and w_{k-1} in shared memory and
// reads the rows next to them from its neighbours' (distributed shared
// memory); one cluster barrier per step, behind which w_{k-1} may be
// overwritten (only w_k is read by others).  No step waits for its sums: the
// threads leave them in shared memory, the ninth warp adds them up during the
// next step and block 0's forms the moments in the one after.  As two launches
// per step, 16 realizations of 64^2 took 18 us a step, 4 of them work: 4725 ->
// 1655 us for 512 moments; now bound by the FP64 pipe (18 operations per node
// and step, lumped) and the barrier.
constexpr int CHEB_CTAS = 8, CHEB_WARPS = 8, CHEB_MAX_N = 128;
template <int SCHEME>
__global__ void __cluster_dims__(CHEB_CTAS, 1, 1) __launch_bounds__(32 * (CHEB_WARPS + 1))
    k_cheb_cluster(const __grid_constant__ DescChunk ch, CoefSrc cs, double a0, double a1, int steps,
                   int K, const double* __restrict__ v, double* __restrict__ mu) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(16) double rowtab[ROW_TABLE];
    __shared__ __align__(16) double psum[2][32 * CHEB_WARPS * 4];   // the threads' sums, by step parity
    __shared__ double slots[2][CHEB_CTAS * 4];   // block 0: the blocks' sums, by step parity
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), b = blockIdx.x / CHEB_CTAS;
    const RDesc& d = ch.d[b];
    if (d.n > CHEB_MAX_N) return;   // the whole cluster: k_cheb
    const int n = d.n, m = n - 1, lg = d.log2n, R = n / CHEB_CTAS, r0 = rank * R;
    const int tid = threadIdx.x, lane = tid & 31;
    const int rows = R * n;
    double2* own = reinterpret_cast<double2*>(smem_raw);   // [2][R][n]
    const double2* above = cl.map_shared_rank(own, (rank + CHEB_CTAS - 1) % CHEB_CTAS) + (R - 1) * n;
    const double2* below = cl.map_shared_rank(own, (rank + 1) % CHEB_CTAS);
    double* slot0 = cl.map_shared_rank(&slots[0][0], 0);
    for (int k = tid; k < rows; k += blockDim.x) {   // v is 8-byte aligned
        const int64_t i = 2 * (d.node_off + (int64_t)r0 * n + k);
        own[k] = make_double2(v[i], v[i + 1]);
    }
    const bool masked = !cs.coef;
    if (masked) fill_row_table<SCHEME>(rowtab, d.a_matrix, d.a_incl);
    // column j, rows i0 .. i1 of the block
    const int groups = 32 * CHEB_WARPS / n, per = max(1, R / groups);
    const int j = tid & m, jm = (j - 1) & m, jp = (j + 1) & m;
    const int i0 = (tid >> lg) * per, i1 = min(R, i0 + per);
    const bool active = tid < 32 * CHEB_WARPS && i0 < R;
    auto cell = [&](int i, int jj) { return cs.cell(d, (r0 + i) & m, jj); };
    unsigned pat = 0;   // masks: two bits per row i0 - 1 .. i1 - 1 (at most nine rows)
    if (active && masked) {
        const uint32_t* mw = cs.mask + d.word_off;
        for (int i = i0 - 1; i < i1; ++i) {
            const int64_t r = (int64_t)((r0 + i) & m) << lg;
            const unsigned x = (mw[(r + jm) >> 5] >> (jm & 31)) & 1u, y = (mw[(r + j) >> 5] >> (j & 31)) & 1u;
            pat |= (x | (y << 1)) << (2 * (i - i0 + 1));
        }
    }
    double mu0 = 0.0, mu1 = 0.0;   // block 0, ninth warp: the first moments
    cl.sync();
    const int summers = n * (R / per);   // threads that hold sums: a multiple of 8
    for (int k = 0; k < steps + 2; ++k) {
        const int cur = (k & 1) * rows, oth = rows - cur;
        if (active && k < steps) {
            double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
            const double f = k == 0 ? 1.0 : 2.0;
            const double f1 = f * a0 / row_scale<SCHEME>(), f2 = f * a1;
            auto rowp = [&](int i) -> const double2* {
                return i < 0 ? above + cur : i >= R ? below + cur : own + cur + i * n;
            };
            const double2* up = rowp(i0 - 1);
            const double2* md = rowp(i0);
            double2 u0 = up[jm], u1 = up[j], u2 = up[jp], c0 = md[jm], c1 = md[j], c2 = md[jp];
            auto row = [&](int i, const StencilRow& w, auto doubled) {
                const double2* dn = rowp(i + 1);
                const double2 d0 = dn[jm], d1 = dn[j], d2 = dn[jp];
                const double2 q = apply_row<SCHEME, decltype(doubled)::value>(w, u0, u1, u2, c0, c1, c2, d0, d1, d2);
                const double2 wm = k == 0 ? make_double2(0.0, 0.0) : own[oth + i * n + j];
                const double2 t = make_double2(fma(f1, q.x, fma(-f2, c1.x, -wm.x)),
                                               fma(f1, q.y, fma(-f2, c1.y, -wm.y)));
                own[oth + i * n + j] = t;
                s0 = fma(c1.x, c1.x, s0);
                s1 = fma(c1.y, c1.y, s1);
                s2 = fma(t.x, c1.x, s2);
                s3 = fma(t.y, c1.y, s3);
                u0 = c0; u1 = c1; u2 = c2;
                c0 = d0; c1 = d1; c2 = d2;
            };
            if (masked) {
                for (int i = i0; i < i1; ++i)
                    row(i, table_row<SCHEME>(rowtab, (pat >> (2 * (i - i0))) & 15u), std::true_type());
            } else {
                RowWalk<SCHEME> walk(cell(i0 - 1, jm), cell(i0 - 1, j));
                for (int i = i0; i < i1; ++i) row(i, walk.step(cell(i, jm), cell(i, j)), std::false_type());
            }
            double2* ps = reinterpret_cast<double2*>(psum[k & 1]) + 2 * tid;
            ps[0] = make_double2(s0, s1);
            ps[1] = make_double2(s2, s3);
        }
        if (tid >= 32 * CHEB_WARPS) {
            // w.w (0, 1) and w'.w (2, 3) of the block, in lanes value, value + 4, ...
            if (k >= 1 && k - 1 < steps) {
                const double* ps = psum[(k - 1) & 1] + lane;
                double x = 0.0, y = 0.0;
                for (int t = 0; t + 16 <= summers; t += 16) {
                    x += ps[4 * t];
                    y += ps[4 * t + 32];
                }
                x += y;
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                if (lane < 4) slot0[((k - 1) & 1) * CHEB_CTAS * 4 + rank * 4 + lane] = x;
            }
            if (rank == 0 && k >= 2) {
                const int q = k - 2;
                double x = slots[q & 1][lane];
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                const double nc = __shfl_down_sync(0xffffffffu, x, 2);   // lanes 0, 1
                if (lane < 2) {
                    double* mb = mu + ((int64_t)b * 2 + lane) * K;
                    if (q == 0) { mu0 = x; mu1 = nc; }
                    if (2 * q < K) mb[2 * q] = q == 0 ? x : 2.0 * x - mu0;
                    if (2 * q + 1 < K) mb[2 * q + 1] = q == 0 ? nc : 2.0 * nc - mu1;
                }
            }
        }
        cl.sync();
    }
}

// Moments of step k from its tile partials, one warp per realization (fixed
// order): mu[b][c][2k] and mu[b][c][2k+1] (k = 0: mu_0 = w_0.w_0, mu_1 = w_1.w_0).
__global__ void k_cheb_moments(const __grid_constant__ DescChunk ch, const double* __restrict__ part,
                               int k, int K, double* __restrict__ mu) {
    const int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (b >= ch.count) return;
    const int t0 = ch.start[b], nt = ch.start[b + 1] - t0;
    if (nt == 0) return;   // a small grid: k_cheb_cluster
    double s[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) s[q] = warp_sum_array(part + (int64_t)t0 * 4 + q, nt, 4);
    if ((threadIdx.x & 31) != 0) return;
    for (int c = 0; c < 2; ++c) {
        double* m = mu + ((int64_t)b * 2 + c) * K;
        const double cc = s[c], nc = s[2 + c];
        const double e = (k == 0) ? cc : 2.0 * cc - m[0];
        const double o = (k == 0) ? nc : 2.0 * nc - m[1];
        if (2 * k < K) m[2 * k] = e;
        if (2 * k + 1 < K) m[2 * k + 1] = o;
    }
}

// ------------------------------------------------------------- adjoint --
// grad[c] = (1/L^2) sum_ij G_ij (xi_i + P_c u_i)^T E (xi_j + P_c u_j): the
// explicit derivative of the energy form (the correctors are stationary).
// E (unit coefficient, K1 (x) M1 + M1 (x) K1) has zero row sums, so
//   x^T E y = sum_{k<l} |E_kl| (x_k - x_l)(y_k - y_l)
// with |E_kl| = w0 - w1 on the four cell edges and 2 w1 on the two
// diagonals: the quadratic forms are built from differences across the cell
// (no cancellation between O(|u|) terms, which would cost up to ~1e-10
// relative accuracy where the local energy is small).
template <int SCHEME>
__global__ void k_backward(const __grid_constant__ DescChunk ch, const double2* __restrict__ u,
                           const double* __restrict__ G, double* __restrict__ grad) {
    const int b = find_real(ch.start, ch.count, blockIdx.x);
    const RDesc& d = ch.d[b];
    const int64_t cell = (int64_t)(blockIdx.x - ch.start[b]) * NODE_TILE + threadIdx.x;
    const int c1 = (int)(cell >> d.log2n), c2 = (int)(cell & (d.n - 1));
    const double2 u00 = ldv(u, d, c1, c2), u01 = ldv(u, d, c1, c2 + 1);
    const double2 u10 = ldv(u, d, c1 + 1, c2), u11 = ldv(u, d, c1 + 1, c2 + 1);
    const double h = d.h;
    const double we = Weights<SCHEME>::w0 - Weights<SCHEME>::w1;   // edges
    const double wd = 2.0 * Weights<SCHEME>::w1;                   // diagonals
    // pairs 00-01, 00-10, 00-11, 01-10, 01-11, 10-11 (second minus first) of
    // v_1 = x_1 + phi_1 = (u00, u01, h + u10, h + u11) and
    // v_2 = x_2 + phi_2 = (u00, h + u01, u10, h + u11)
    const double d1[6] = {u01.x - u00.x,       h + (u10.x - u00.x), h + (u11.x - u00.x),
                          h + (u10.x - u01.x), h + (u11.x - u01.x), u11.x - u10.x};
    const double d2[6] = {h + (u01.y - u00.y), u10.y - u00.y,       h + (u11.y - u00.y),
                          (u10.y - u01.y) - h, u11.y - u01.y,       h + (u11.y - u10.y)};
    const double w[6] = {we, we, wd, wd, we, we};
    double e11 = 0.0, e12 = 0.0, e22 = 0.0;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        e11 = fma(w[k] * d1[k], d1[k], e11);
        e12 = fma(w[k] * d1[k], d2[k], e12);
        e22 = fma(w[k] * d2[k], d2[k], e22);
    }
    const double* Gb = G + 4 * (int64_t)b;   // G is offset to the chunk's first realization
    grad[d.node_off + cell] = d.inv_vol * (Gb[0] * e11 + (Gb[1] + Gb[2]) * e12 + Gb[3] * e22);
}

// ---------------------------------------------------------------- A_hom --
// Cell-form partial sums and the final reduction (rve_ahom.cuh).
// Mixed solves: one block per strip (a_hom_strip).
template <int SCHEME>
__global__ void __launch_bounds__(256, 3)
    k_a_hom_strip(const RDesc* __restrict__ desc, const int32_t* __restrict__ start, int batch,
                  CoefSrc cs, const double2* __restrict__ u, double* __restrict__ part) {
    __shared__ double red[64];
    __shared__ float sc[5];
    const int b = find_real(start, batch, blockIdx.x);
    const RDesc d = desc[b];
    a_hom_strip<SCHEME>(d, blockIdx.x - start[b], cs, u, red, sc,
                        part + (int64_t)blockIdx.x * AHOM_NP);
}

// FP64 solves: double-double partials (16 doubles per tile), of the energy
// form alone or of both forms.
template <int SCHEME, bool FLUX>
__global__ void __launch_bounds__(256) k_a_hom_part_dd(const RDesc* __restrict__ desc,
                                                       const int32_t* __restrict__ start, int batch,
                                                       CoefSrc cs,
                                                       const double2* __restrict__ u,
                                                       double* __restrict__ part) {
    __shared__ ddouble red[8 * (FLUX ? AHOM_NP : 4)];
    const int b = find_real(start, batch, blockIdx.x);
    const RDesc d = desc[b];
    const int cells = a_hom_cells(d.n);
    double* out = part + (int64_t)blockIdx.x * 2 * AHOM_NP;
    a_hom_tile_dd<SCHEME, FLUX>(d, blockIdx.x - start[b], cells, cs, u, red, out);
}

template <int SCHEME>
__global__ void __launch_bounds__(256) k_a_hom_final_dd(const RDesc* __restrict__ desc,
                                                        const int32_t* __restrict__ start,
                                                        const double* __restrict__ part,
                                                        double* __restrict__ A,
                                                        double* __restrict__ Alo,
                                                        double* __restrict__ Af) {
    __shared__ ddouble red[AHOM_NP];
    const int b = blockIdx.x;
    const RDesc d = desc[b];
    a_hom_finish_dd<SCHEME>(d, part + (int64_t)start[b] * 2 * AHOM_NP, start[b + 1] - start[b], red,
                            A + 4 * (int64_t)b, Alo ? Alo + 4 * (int64_t)b : nullptr,
                            Af ? Af + 4 * (int64_t)b : nullptr);
}

// One warp per realization.
template <int SCHEME>
__global__ void k_a_hom_final(const RDesc* __restrict__ desc, const int32_t* __restrict__ start,
                              int batch, const double* __restrict__ part, double* __restrict__ A,
                              double* __restrict__ Af) {
    const int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (b >= batch) return;
    const RDesc d = desc[b];
    a_hom_finish<SCHEME>(d, part + (int64_t)start[b] * AHOM_NP, start[b + 1] - start[b],
                         A + 4 * (int64_t)b, Af ? Af + 4 * (int64_t)b : nullptr);
}

// ------------------------------------------------------------- launchers --
// Splits the plan's realizations into chunks and calls `fn(chunk, first)`
// with start[] = prefix sums of units(d) over the chunk.
template <typename UnitsFn, typename LaunchFn>
static cudaError_t for_chunks(const Plan& p, UnitsFn units, LaunchFn fn) {
    for (int b0 = 0; b0 < p.batch; b0 += CHUNK) {
        DescChunk ch;
        ch.count = std::min(CHUNK, p.batch - b0);
        ch.start[0] = 0;
        for (int k = 0; k < ch.count; ++k) {
            ch.d[k] = p.desc[b0 + k];
            ch.start[k + 1] = ch.start[k] + (int32_t)units(ch.d[k]);
        }
        for (int k = ch.count + 1; k <= CHUNK; ++k) ch.start[k] = ch.start[ch.count];
        cudaError_t e = fn(ch, b0);
        if (e != cudaSuccess) return e;
        note_launch();
    }
    return cudaSuccess;
}

cudaError_t launch_gen_field(const Plan& p, void* /*ws*/, uint32_t* mask, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(mask, 0, sizeof(uint32_t) * (size_t)p.words, s);
    if (e != cudaSuccess) return e;
    return for_chunks(p, [](const RDesc& d) { return (int64_t)d.n_incl * d.s; },
                      [&](const DescChunk& ch, int) {
                          const int total = ch.start[ch.count];
                          if (total == 0) return cudaSuccess;
                          k_gen_field<<<(total + 255) / 256, 256, 0, s>>>(ch, mask);
                          return cudaGetLastError();
                      });
}

static int64_t node_tiles(const RDesc& d) { return ((int64_t)d.n * d.n) / NODE_TILE; }

cudaError_t launch_rhs(const Plan& p, void*, const uint32_t* mask, const double* coef, double* f,
                       cudaStream_t s) {
    CoefSrc cs{mask, coef};
    return for_chunks(p, node_tiles, [&](const DescChunk& ch, int) {
        k_rhs<<<ch.start[ch.count], NODE_TILE, 0, s>>>(ch, cs, reinterpret_cast<double2*>(f));
        return cudaGetLastError();
    });
}

cudaError_t launch_coef_from_mask(const Plan& p, const uint32_t* mask, double* coef,
                                  cudaStream_t s) {
    return for_chunks(p, node_tiles, [&](const DescChunk& ch, int) {
        k_coef_from_mask<<<ch.start[ch.count], NODE_TILE, 0, s>>>(ch, mask, coef);
        return cudaGetLastError();
    });
}

cudaError_t launch_stiffness(const Plan& p, void*, const uint32_t* mask, const double* coef,
                             int scheme, int precision, const void* x, void* y, cudaStream_t s) {
    CoefSrc cs{mask, coef};
    // rows per thread: 16, fewer while that leaves under four blocks per SM
    auto launch = [&]<typename V>(const V* xx, V* yy) {
        const bool pairs = ((reinterpret_cast<uintptr_t>(xx) | reinterpret_cast<uintptr_t>(yy)) & 15) == 0;
        int rows = 16;
        while (rows > 2 && p.nodes < (int64_t)rows * STIFF_THREADS * (int64_t)(16 / sizeof(V)) * 4 * 152) rows /= 2;
        return for_chunks(p,
                          [&](const RDesc& d) {
                              return (int64_t)(d.n / stiff_cols<V>(d.n)) * (d.n / stiff_block_rows<V>(d.n, rows));
                          },
                          [&](const DescChunk& ch, int) {
                              const int g = ch.start[ch.count];
                              if (scheme == RVE_Q1_LUMPED) k_stiffness<1, V><<<g, STIFF_THREADS, 0, s>>>(ch, cs, xx, yy, rows, pairs);
                              else k_stiffness<0, V><<<g, STIFF_THREADS, 0, s>>>(ch, cs, xx, yy, rows, pairs);
                              return cudaGetLastError();
                          });
    };
    if (precision == RVE_FP64)
        return launch(static_cast<const double2*>(x), static_cast<double2*>(y));
    return launch(static_cast<const float2*>(x), static_cast<float2*>(y));
}

cudaError_t launch_mass(const Plan& p, int scheme, const double* x, double* y, cudaStream_t s) {
    return for_chunks(p, node_tiles, [&](const DescChunk& ch, int) {
        const int g = ch.start[ch.count];
        const double2* xx = reinterpret_cast<const double2*>(x);
        double2* yy = reinterpret_cast<double2*>(y);
        if (scheme == RVE_Q1_LUMPED) k_mass<1><<<g, NODE_TILE, 0, s>>>(ch, xx, yy);
        else k_mass<0><<<g, NODE_TILE, 0, s>>>(ch, xx, yy);
        return cudaGetLastError();
    });
}

size_t cheb_workspace_size(const Plan& p) {
    int64_t tiles = 0;   // most node tiles of any launch chunk
    for (int b0 = 0; b0 < p.batch; b0 += CHUNK) {
        int64_t t = 0;
        for (int k = b0; k < std::min(p.batch, b0 + CHUNK); ++k)
            t += ((int64_t)p.desc[k].n * p.desc[k].n) / NODE_TILE;
        tiles = std::max(tiles, t);
    }
    auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
    return 2 * up(sizeof(double2) * (size_t)p.nodes) + up(sizeof(double) * 4 * (size_t)tiles);
}

cudaError_t launch_cheb(const Plan& p, void* ws, const uint32_t* mask, const double* coef,
                        int scheme, const double* v, int K, double lo, double hi, double* mu,
                        cudaStream_t s) {
    auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
    char* w = static_cast<char*>(ws);
    double2* wa = reinterpret_cast<double2*>(w);
    double2* wb = reinterpret_cast<double2*>(w + up(sizeof(double2) * (size_t)p.nodes));
    double* part = reinterpret_cast<double*>(w + 2 * up(sizeof(double2) * (size_t)p.nodes));
    const double a0 = 2.0 / (hi - lo), a1 = (hi + lo) / (hi - lo);
    CoefSrc cs{mask, coef};
    const int steps = (K + 1) / 2;
    const size_t most = 2 * sizeof(double2) * CHEB_MAX_N * CHEB_MAX_N / CHEB_CTAS;
    cudaError_t e = cudaFuncSetAttribute(k_cheb_cluster<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_cheb_cluster<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    if (e != cudaSuccess) return e;
    // the form by each grid's own size (the two round differently)
    auto step_tiles = [](const RDesc& d) { return d.n <= CHEB_MAX_N ? (int64_t)0 : node_tiles(d); };
    return for_chunks(p, step_tiles, [&](const DescChunk& ch, int first_real) {
        double* m = mu + (int64_t)first_real * 2 * K;
        int maxn = 0;
        for (int k = 0; k < ch.count; ++k)
            if (ch.d[k].n <= CHEB_MAX_N) maxn = std::max(maxn, ch.d[k].n);
        if (maxn > 0) {   // two vectors of a realization fit a cluster's shared memory
            const size_t smem = 2 * sizeof(double2) * (size_t)maxn * maxn / CHEB_CTAS;
            auto kern = scheme == RVE_Q1_LUMPED ? k_cheb_cluster<1> : k_cheb_cluster<0>;
            kern<<<ch.count * CHEB_CTAS, 32 * (CHEB_WARPS + 1), smem, s>>>(ch, cs, a0, a1, steps, K, v, m);
            const cudaError_t ce = cudaGetLastError();
            if (ce != cudaSuccess) return ce;
        }
        for (int k = 0; k < ch.count;) {   // w_0 of every run of large grids
            int e = k;
            while (e < ch.count && ch.d[e].n > CHEB_MAX_N) ++e;
            if (e > k) {
                const int64_t from = ch.d[k].node_off;
                const int64_t to = ch.d[e - 1].node_off + (int64_t)ch.d[e - 1].n * ch.d[e - 1].n;
                const cudaError_t ce = cudaMemcpyAsync(wb + from, v + 2 * from, sizeof(double2) * (size_t)(to - from),
                                                       cudaMemcpyDeviceToDevice, s);
                if (ce != cudaSuccess) return ce;
            }
            k = e + 1;
        }
        if (ch.start[ch.count] == 0) return cudaSuccess;
        const int g = ch.start[ch.count];
        double2* cur = wb;    // w_k
        double2* oth = wa;    // in: w_{k-1}, out: w_{k+1}
        for (int k = 0; k < steps; ++k) {
            if (scheme == RVE_Q1_LUMPED)
                k_cheb<1><<<g, NODE_TILE, 0, s>>>(ch, cs, a0, a1, k == 0, cur, oth, part);
            else
                k_cheb<0><<<g, NODE_TILE, 0, s>>>(ch, cs, a0, a1, k == 0, cur, oth, part);
            k_cheb_moments<<<(ch.count + 7) / 8, 256, 0, s>>>(ch, part, k, K, m);
            note_launch(2);
            const cudaError_t le = cudaGetLastError();
            if (le != cudaSuccess) return le;
            std::swap(cur, oth);
        }
        return cudaSuccess;
    });
}

cudaError_t launch_backward(const Plan& p, void*, int scheme, const double* u, const double* gradA,
                            double* grad_coef, cudaStream_t s) {
    return for_chunks(p, node_tiles, [&](const DescChunk& ch, int first) {
        const double* G = gradA + 4 * (int64_t)first;
        const double2* uu = reinterpret_cast<const double2*>(u);
        const int g = ch.start[ch.count];
        if (scheme == RVE_Q1_LUMPED) k_backward<1><<<g, NODE_TILE, 0, s>>>(ch, uu, G, grad_coef);
        else k_backward<0><<<g, NODE_TILE, 0, s>>>(ch, uu, G, grad_coef);
        return cudaGetLastError();
    });
}

cudaError_t launch_a_hom(const Plan& p, void* ws, const uint32_t* mask, const double* coef,
                         int scheme, int precision, const double* u, double* A, double* A_lo,
                         double* A_flux, cudaStream_t s) {
    char* w = static_cast<char*>(ws);
    const RDesc* desc = reinterpret_cast<const RDesc*>(w + p.o_desc);
    const int32_t* start = reinterpret_cast<const int32_t*>(w + p.o_startA);
    double* part = reinterpret_cast<double*>(w + p.o_partA);
    CoefSrc cs{mask, coef};
    const double2* uu = reinterpret_cast<const double2*>(u);
    const bool lumped = scheme == RVE_Q1_LUMPED;
    const int gf = (p.batch + 7) / 8;
    if (precision == RVE_FP64) {
        auto parts = lumped ? (A_flux ? k_a_hom_part_dd<1, true> : k_a_hom_part_dd<1, false>)
                            : (A_flux ? k_a_hom_part_dd<0, true> : k_a_hom_part_dd<0, false>);
        parts<<<p.tilesA, p.threadsA, 0, s>>>(desc, start, p.batch, cs, uu, part);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        if (lumped) k_a_hom_final_dd<1><<<p.batch, 256, 0, s>>>(desc, start, part, A, A_lo, A_flux);
        else k_a_hom_final_dd<0><<<p.batch, 256, 0, s>>>(desc, start, part, A, A_lo, A_flux);
    } else {
        const int32_t* start2 = reinterpret_cast<const int32_t*>(w + p.o_startA2);
        if (lumped) k_a_hom_strip<1><<<p.tilesA2, 256, 0, s>>>(desc, start2, p.batch, cs, uu, part);
        else k_a_hom_strip<0><<<p.tilesA2, 256, 0, s>>>(desc, start2, p.batch, cs, uu, part);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        if (lumped) k_a_hom_final<1><<<gf, 256, 0, s>>>(desc, start2, p.batch, part, A, A_flux);
        else k_a_hom_final<0><<<gf, 256, 0, s>>>(desc, start2, p.batch, part, A, A_flux);
    }
    note_launch(2);
    return cudaGetLastError();
}

}  // namespace rve
