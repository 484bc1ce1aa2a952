// rve_pipeline.cuh -- device code of the preconditioned CG for the two corrector problems
// (Sec. 3.4 and 4.1), batched over realizations, on sm_103a.
//
// Preconditioner (Sec. 3.4): B = c0 A_Delta + delta I with A_Delta the
// periodic 5-point Laplacian.  On the torus B is diagonalised by the
// separable real Hartley transform H (x) H, (H (x) H)^2 = n^2 I, so
//   B^{-1} r = (H (x) H) diag(1 / (n^2 sigma)) (H (x) H) r,
//   sigma(k1,k2) = c0 (4 sin^2(pi k1/n) + 4 sin^2(pi k2/n)) + delta,
// the constant mode being dropped when delta = 0.  Each 1D Hartley pass
// transforms the two correctors at once: the complex DFT of (r_1 + i r_2)
// along the axis is split into H r_1 and H r_2 (see hartley_pair).  Since
// the transform is orthogonal up to n, r.z = (1/n^2) sum (H(x)H r)^2 / sigma
// is read off in the transform domain.
//
// Fused pipeline (one CG step = three passes over the vectors, R or S first,
// + a control kernel; both correctors of a realization travel together as a pair):
//   R  (REFINE steps only) r64 = f - A(u + s (x + alpha p)), the true
//      residual in double words (FP64 for the FP64 path), partial |r64|^2
//   S  z = inverse row-Hartley(zhat) on the tile + halo rows, p_new = z +
//      beta p_old, x += alpha_prev p_old (the solution update lags one
//      step), q = A p_new, partial p.q; the last block of a realization
//      forms alpha = rho / p.q
//   U  rt -= alpha H q (the residual kept as its row transform rt = H r),
//      partial |r|^2 = |rt|^2 / n (REFINE: u += s (x + alpha p), x = 0,
//      rt = H (r64 / |r64|))
//   C  periodic tridiagonal solve along every column of rt (the row
//      transform diagonalises the row factor of A_Delta), scaled, into
//      zhat; partial rho = r.z
//   K  per realization: reduce the partials in a fixed order, set alpha,
//      beta, convergence and the next phase.
// In MIXED precision x, rt, q, zhat, p are float2 and u is the double-word
// iterate: every REFINE step recomputes the true residual in double words
// and restarts the FP32 inner iteration on the scaled residual equation
// (iterative refinement).
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "rve_colsolve.cuh"
#include "rve_common.cuh"
#include "rve_internal.h"

namespace rve {

// Control words (int32) in the workspace: [0] realizations done, then the
// persistent kernel's grid barrier.
enum { CTL_ARRIVE = 8, CTL_GEN = 9, CTL_ERR = 10, CTL_GROUPS = 11 };

struct Ctx {
    int batch;
    const RDesc* __restrict__ desc;
    const int32_t* __restrict__ startS;
    const int32_t* __restrict__ startU;
    const int32_t* __restrict__ startC;
    // written during a solve (by other blocks of the persistent launch too):
    // no __restrict__, so that every read is a coherent load
    RState* st;
    double* partS;
    double* partU;
    double* partC;
    double* uscal;     // [batch][4]: the update kernel's step scalars and the sums (see finish_S)
    int* tiles_done;   // [batch]: stencil/refine blocks finished this step
    Tables tb;
    CoefSrc cs;
    double2* u;
    void* X;
    void* R;
    void* Q;
    void* T;
    void* P0;
    void* P1;
    double tol, inner_tol, delta;
    int max_iter;
    int* ndone;
};

// ---------------------------------------------------------- row helpers --
// y + (ax, ay) * x componentwise; the scalars are already in the vector's
// type (no per-element conversion: on GB300 conversions from double run on
// the slow FP64 pipe).
template <typename V>
__device__ __forceinline__ V axpy2(V y, typename ScalarOf<V>::T ax, typename ScalarOf<V>::T ay, V x) {
    V r;
    r.x = y.x + ax * x.x;
    r.y = y.y + ay * x.y;
    return r;
}

template <typename V>
__device__ __forceinline__ int64_t node_of(const RDesc& d, int row, int col) {
    return d.node_off + ((int64_t)row << d.log2n) + col;
}

// Thread layout of the row kernels: T = n/8 threads per row, so
// blockDim/T rows per group; qq = row within the group, t = thread within
// row.  With a compile-time size (LOG2N > 0) T and the divisions fold.
template <int LOG2N>
struct RowLayout {
    Sz<LOG2N> z;
    int qq, t, G;
    __device__ __forceinline__ explicit RowLayout(int log2n) : z(log2n) {
        G = blockDim.x / z.T;
        qq = threadIdx.x / z.T;
        t = threadIdx.x - qq * z.T;
    }
};

template <int LOG2N>
__device__ __forceinline__ int64_t node_at(const RDesc& d, const Sz<LOG2N>& z, int row, int col) {
    return d.node_off + ((int64_t)row << z.log2n) + col;
}

// Calls body.template operator()<LOG2N>() with the realization's size as a
// compile-time constant (n = 32 .. 2048).
template <typename F>
__device__ __forceinline__ void dispatch_size(int log2n, F&& body) {
    switch (log2n) {
        case 5: body.template operator()<5>(); break;
        case 6: body.template operator()<6>(); break;
        case 7: body.template operator()<7>(); break;
        case 8: body.template operator()<8>(); break;
        case 9: body.template operator()<9>(); break;
        case 10: body.template operator()<10>(); break;
        default: body.template operator()<11>(); break;
    }
}

// ----------------------------------------------------------- S kernel --
template <typename V>
__device__ __forceinline__ double2 refine_w(const Ctx& c, const RDesc& d, const RState& s, int i,
                                            int j, const V* P) {
    const int64_t node = d.node_off + ((int64_t)(i & (d.n - 1)) << d.log2n) + (j & (d.n - 1));
    const double2 uu = c.u[node];
    const double2 xx = to_d2(static_cast<const V*>(c.X)[node]);
    const double2 pp = to_d2(P[node]);
    return make_double2(uu.x + s.s[0] * (xx.x + s.alpha[0] * pp.x),
                        uu.y + s.s[1] * (xx.y + s.alpha[1] * pp.y));
}

// Cell value from the shared-memory mask rows of the tile (cell rows
// r0-1 .. r0+TR-1 stored at mrow 0 .. TR) or from the coefficient array.
template <typename T>
struct TileCoef {
    const uint32_t* mrows;   // shared, (TR+1) x (n/32) words, or null
    int wpr;                 // words per row
    T a_incl, a_matrix;      // the two values in the arithmetic type
    __device__ __forceinline__ T cell(const CoefSrc& cs, const RDesc& d, int mrow, int c1,
                                      int c2) const {
        if (mrows) {
            const uint32_t w = mrows[mrow * wpr + (c2 >> 5)];
            return ((w >> (c2 & 31)) & 1u) ? a_incl : a_matrix;
        }
        return (T)cs.cell(d, c1 & (d.n - 1), c2);
    }
};

// Called by every stencil/refine block after it wrote its partial sums of
// realization b.  The block that finishes last (atomic tile counter) sums
// all of them in tile order -- deterministic whichever block is last -- and
// stores the update kernel's scalars: in ITER alpha = rho / p.q (0 for a
// frozen corrector), in REFINE 1/|r64| (0 once the corrector meets the
// tolerance).  The update kernel then starts without any FP64 work.
inline __device__ void finish_S(const Ctx& c, int b, const RState& s, bool refine, double scale) {
    __shared__ int last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const int nt = c.startS[b + 1] - c.startS[b];
        last = (atomicAdd(c.tiles_done + b, 1) == nt - 1);
    }
    __syncthreads();
    if (!last) return;
    if (threadIdx.x < 64) {   // one warp per corrector
        __threadfence();
        const int k = threadIdx.x >> 5;
        const int t0 = c.startS[b], nt = c.startS[b + 1] - t0;
        const double sum = warp_sum_array(c.partS + 2 * (int64_t)t0 + k, nt, 2);
        if ((threadIdx.x & 31) == 0) {
            double a;
            if (!refine) {
                a = s.active[k] ? s.rho[k] / sum : 0.0;
                c.uscal[4 * b + 2 + k] = scale * a;
            } else {
                const double rn = sqrt(sum);
                const bool conv = (s.refinements == 0) ? (rn == 0.0) : (rn <= c.tol * s.fnorm[k]);
                a = conv ? 0.0 : 1.0 / rn;
                c.uscal[4 * b + 2 + k] = sum;
            }
            c.uscal[4 * b + k] = a;
            if (k == 0) c.tiles_done[b] = 0;   // ready for the next step
        }
    }
}

// Mixed path: the FP64-accurate iterate lives in the caller's u buffer as a
// double word per node and corrector (float4 = hi.x, hi.y, lo.x, lo.y) until
// the solve ends (k_u_finalize).  The refine and update kernels both form
// the new iterate w = u + s (x + alpha p) with this function -- correction
// in FP32, added to u as a double word -- so that the residual computed for
// w belongs to exactly the w that is stored.
struct DWScal { float sx, sy, ax, ay; };
__device__ __forceinline__ float4 w_new(float4 u, float2 x, float2 p, const DWScal& k) {
    const float dx = __fmul_rn(k.sx, __fmaf_rn(k.ax, p.x, x.x));
    const float dy = __fmul_rn(k.sy, __fmaf_rn(k.ay, p.y, x.y));
    const dword wx = dw_add(dword{u.x, u.z}, dx);
    const dword wy = dw_add(dword{u.y, u.w}, dy);
    return make_float4(wx.hi, wy.hi, wx.lo, wy.lo);
}


// REFINE step of the mixed path: r = f - A w for the tile's rows with
// w = u + s (x + alpha p), in double-word arithmetic on the FP32 pipe (no
// FP64 per node).  The stiffness and the right-hand side are scaled by
// K = 6 (consistent) resp. 2 (lumped) so that every stencil weight is an
// integer multiple of a cell value: K A has centre 2 K w0 (sum of the four
// cells), edges -(sum of the two shared cells), corners -2 K w1 (shared
// cell), and K f_1 = (K h/2)(a_0m + a_00 - a_mm - a_m0).  r_K = K f - K A w
// is accumulated as a compensated dot product, so its absolute error is
// O(eps_32^2) times the size of the stencil terms -- far below the outer
// tolerance -- and r = r_K / K is rounded to FP32 (the inner iteration's
// type).  Each thread walks down one column with a 3 x 3 window of w.
// EXACT: both cell values are integers of magnitude <= 2^20 (the paper's
// two-valued coefficients 1 and the contrast), so every cell sum and scaled
// weight below is exact in one float; the weights are then floats (CW)
// instead of double words, with the same values and so the same results.
template <int SCHEME, bool EXACT>
__device__ void refine_tile_dw(const Ctx& c, int tile, int b, const RState& s, const RDesc& d) {
    typedef std::conditional_t<EXACT, float, dword> CW;
    __shared__ double red[64];
    __shared__ float sc[9];
    const int n = d.n;
    const int r0 = (tile - c.startS[b]) * d.tS;
    const int rows = min(d.tS, n - r0);   // the last tile may be shorter
    if (threadIdx.x == 0) {
        sc[0] = (float)s.s[0];
        sc[1] = (float)s.s[1];
        sc[2] = (float)s.alpha[0];
        sc[3] = (float)s.alpha[1];
        const dword ai = dw_of(d.a_incl), am = dw_of(d.a_matrix);
        sc[4] = ai.hi; sc[5] = ai.lo; sc[6] = am.hi; sc[7] = am.lo;
        sc[8] = (float)d.h;   // 1/m0, a power of two: exact
    }
    __syncthreads();
    const DWScal k{sc[0], sc[1], sc[2], sc[3]};
    const dword aI{sc[4], sc[5]}, aM{sc[6], sc[7]};
    const bool first = (s.refinements == 0);   // u = x = p = 0: r = f
    constexpr float CEN = SCHEME == 0 ? 4.f : 2.f;      // 2 K w0
    constexpr float COR = SCHEME == 0 ? 2.f : 0.f;      // 2 K w1
    constexpr float KH = SCHEME == 0 ? 3.f : 1.f;       // K / 2
    constexpr float INVK = SCHEME == 0 ? (1.f / 6.f) : 0.5f;
    const float kh2 = KH * sc[8];   // K h / 2: exact
    const float4* U = reinterpret_cast<const float4*>(c.u);
    const float2* X = static_cast<const float2*>(c.X);
    const float2* P = static_cast<const float2*>(s.parity ? c.P1 : c.P0);
    float2* Q = static_cast<float2*>(c.Q);
    auto wat = [&](int i, int j) -> float4 {
        if (first) return make_float4(0.f, 0.f, 0.f, 0.f);
        const int64_t node = d.node_off + ((int64_t)(i & (n - 1)) << d.log2n) + (j & (n - 1));
        return w_new(U[node], X[node], P[node], k);
    };
    auto cell = [&](int i, int j) -> CW {
        const int64_t ci = ((int64_t)(i & (n - 1)) << d.log2n) + (j & (n - 1));
        if constexpr (EXACT) {   // mask only (no explicit coefficients)
            const uint32_t w = __ldg(c.cs.mask + d.word_off + (ci >> 5));
            return ((w >> (ci & 31)) & 1u) ? aI.hi : aM.hi;
        } else {
            if (c.cs.coef) return dw_of(__ldg(c.cs.coef + d.node_off + ci));
            const uint32_t w = __ldg(c.cs.mask + d.word_off + (ci >> 5));
            return ((w >> (ci & 31)) & 1u) ? aI : aM;
        }
    };
    // cell-weight arithmetic in CW: exact float operations, or double words
    auto wadd = [](CW x, CW y) -> CW {
        if constexpr (EXACT) return __fadd_rn(x, y); else return dw_add(x, y);
    };
    auto wsub = [](CW x, CW y) -> CW {
        if constexpr (EXACT) return __fsub_rn(x, y); else return dw_add(x, dw_neg(y));
    };
    auto wscale2 = [](CW x, float p2) -> CW {
        if constexpr (EXACT) return x * p2; else return dw_scale2(x, p2);
    };
    auto wmulf = [](CW x, float f) -> dword {
        if constexpr (EXACT) {
            const float p = __fmul_rn(x, f);
            return {p, __fmaf_rn(x, f, -p)};
        } else {
            return dw_mulf(x, f);
        }
    };
    dword nx{0.f, 0.f}, ny{0.f, 0.f};   // |r|^2, double-word per thread
    // n < 256: 256 / n groups of threads share the tile's rows
    const int W = min(n, (int)blockDim.x), per = (rows + (int)blockDim.x / W - 1) / ((int)blockDim.x / W);
    const int q0 = ((int)threadIdx.x / W) * per, q1 = min(rows, q0 + per);
    const int col = q0 < q1 ? (int)threadIdx.x & (W - 1) : n;
    if (first) {   // u = x = p = 0: r = f, the same arithmetic without the zero terms
        for (int j = col; j < n; j += blockDim.x) {
            CW cmm = cell(r0 + q0 - 1, j - 1), cm0 = cell(r0 + q0 - 1, j);
            for (int q = q0; q < q1; ++q) {
                const int i = r0 + q;
                const CW c0m = cell(i, j - 1), c00 = cell(i, j);
                dword kfx, kfy;   // K f
                if (c.cs.f) {
                    const double2 fl = c.cs.f[d.node_off + ((int64_t)i << d.log2n) + j];
                    kfx = dw_mulf(dw_split(fl.x), 2.f * KH);
                    kfy = dw_mulf(dw_split(fl.y), 2.f * KH);
                } else {
                    const CW top = wadd(cmm, cm0), bot = wadd(c0m, c00);
                    const CW lft = wadd(cmm, c0m), rgt = wadd(cm0, c00);
                    kfx = wmulf(wsub(bot, top), kh2);
                    kfy = wmulf(wsub(rgt, lft), kh2);
                }
                const DotDW rx(kfx), ry(kfy);
                const float2 r = make_float2(rx.value() * INVK, ry.value() * INVK);
                Q[d.node_off + ((int64_t)i << d.log2n) + j] = r;
                nx = dw_add(nx, r.x * r.x);
                ny = dw_add(ny, r.y * r.y);
                cmm = c0m; cm0 = c00;
            }
        }
    }
    for (int j = first ? n : col; j < n; j += blockDim.x) {
        const int ra = r0 + q0 - 1;
        float4 a0 = wat(ra, j - 1), a1 = wat(ra, j), a2 = wat(ra, j + 1);
        float4 b0 = wat(ra + 1, j - 1), b1 = wat(ra + 1, j), b2 = wat(ra + 1, j + 1);
        CW cmm = cell(ra, j - 1), cm0 = cell(ra, j);
        for (int q = q0; q < q1; ++q) {
            const int i = r0 + q;
            const float4 e0 = wat(i + 1, j - 1), e1 = wat(i + 1, j), e2 = wat(i + 1, j + 1);
            const CW c0m = cell(i, j - 1), c00 = cell(i, j);
            const CW top = wadd(cmm, cm0);   // cells shared with (i-1, j)
            const CW bot = wadd(c0m, c00);   // with (i+1, j)
            const CW lft = wadd(cmm, c0m);   // with (i, j-1)
            const CW rgt = wadd(cm0, c00);   // with (i, j+1)
            const CW cen = wscale2(wadd(top, bot), -CEN);
            dword kfx, kfy;   // K f
            if (c.cs.f) {
                const double2 fl = c.cs.f[d.node_off + ((int64_t)i << d.log2n) + j];
                kfx = dw_mulf(dw_split(fl.x), 2.f * KH);
                kfy = dw_mulf(dw_split(fl.y), 2.f * KH);
            } else {
                kfx = wmulf(wsub(bot, top), kh2);
                kfy = wmulf(wsub(rgt, lft), kh2);
            }
            DotDW rx(kfx), ry(kfy);
            rx.add(cen, b1.x, b1.z); ry.add(cen, b1.y, b1.w);
            rx.add(top, a1.x, a1.z); ry.add(top, a1.y, a1.w);
            rx.add(bot, e1.x, e1.z); ry.add(bot, e1.y, e1.w);
            rx.add(lft, b0.x, b0.z); ry.add(lft, b0.y, b0.w);
            rx.add(rgt, b2.x, b2.z); ry.add(rgt, b2.y, b2.w);
            if (COR != 0.f) {
                const CW kmm = wscale2(cmm, COR), km0 = wscale2(cm0, COR);
                const CW k0m = wscale2(c0m, COR), k00 = wscale2(c00, COR);
                rx.add(kmm, a0.x, a0.z); ry.add(kmm, a0.y, a0.w);
                rx.add(km0, a2.x, a2.z); ry.add(km0, a2.y, a2.w);
                rx.add(k0m, e0.x, e0.z); ry.add(k0m, e0.y, e0.w);
                rx.add(k00, e2.x, e2.z); ry.add(k00, e2.y, e2.w);
            }
            const float2 r = make_float2(rx.value() * INVK, ry.value() * INVK);
            Q[d.node_off + ((int64_t)i << d.log2n) + j] = r;
            nx = dw_add(nx, r.x * r.x);
            ny = dw_add(ny, r.y * r.y);
            a0 = b0; a1 = b1; a2 = b2;
            b0 = e0; b1 = e1; b2 = e2;
            cmm = c0m; cm0 = c00;
        }
    }
    DotAcc<float> ax, ay;
    ax.hi = nx.hi; ax.lo = nx.lo;
    ay.hi = ny.hi; ay.lo = ny.lo;
    double sx = 0.0, sy = 0.0;
    block_sum2(ax, ay, red, sx, sy);
    if (threadIdx.x == 0) {
        c.partS[2 * (int64_t)tile] = sx;
        c.partS[2 * (int64_t)tile + 1] = sy;
    }
    finish_S(c, b, s, true, 1.0);
}

// REFINE step: r64 = f - A(u + s (x + alpha p)) for the tile's rows, stored
// (rounded to the vector type) in q, partial |r64|^2 into partS -- in FP64
// for the FP64 path, in double words for the mixed path (refine_tile_dw).
template <int SCHEME>
__device__ void refine_tile_fp64(const Ctx& c, int tile, int b, const RState& s, const RDesc& d) {
    typedef double2 V;
    __shared__ double red[64];
    const int n = d.n;
    const int r0 = (tile - c.startS[b]) * d.tS;
    const int rows = min(d.tS, n - r0);   // the last tile may be shorter
    const V* Pold = static_cast<const V*>(s.parity ? c.P1 : c.P0);
    V* Q = static_cast<V*>(c.Q);
    const bool first = (s.refinements == 0);   // u = x = p = 0: r = f
    DotAcc<double> a64x, a64y;   // exact FP64 |r64|^2
    for (int idx = threadIdx.x; idx < rows * n; idx += blockDim.x) {
        const int i = r0 + (idx >> d.log2n), j = idx & (n - 1);
        const Cells4 a = cells_at(c.cs, d, i, j);
        const double2 f = load_at(c.cs, d, ((int64_t)i << d.log2n) + j, a);
        double2 Aw = make_double2(0.0, 0.0);
        constexpr double IK = 1.0 / row_scale<SCHEME>();
        if (!first)
            Aw = apply_row<SCHEME, false>(
                RowWalk<SCHEME>(a.mm, a.m0).step(a.z0m, a.z00), refine_w(c, d, s, i - 1, j - 1, Pold), refine_w(c, d, s, i - 1, j, Pold),
                refine_w(c, d, s, i - 1, j + 1, Pold), refine_w(c, d, s, i, j - 1, Pold),
                refine_w(c, d, s, i, j, Pold), refine_w(c, d, s, i, j + 1, Pold),
                refine_w(c, d, s, i + 1, j - 1, Pold), refine_w(c, d, s, i + 1, j, Pold),
                refine_w(c, d, s, i + 1, j + 1, Pold));
        const double2 r64 = make_double2(fma(-IK, Aw.x, f.x), fma(-IK, Aw.y, f.y));
        Q[node_of<V>(d, i, j)] = from_d2<V>(r64);
        a64x.add(r64.x, r64.x);
        a64y.add(r64.y, r64.y);
    }
    double sx = 0.0, sy = 0.0;
    block_sum2(a64x, a64y, red, sx, sy);
    if (threadIdx.x == 0) {
        c.partS[2 * (int64_t)tile] = sx;
        c.partS[2 * (int64_t)tile + 1] = sy;
    }
    finish_S(c, b, s, true, 1.0);
}

template <typename V, int SCHEME>
__device__ __forceinline__ void refine_tile(const Ctx& c, int tile, int b, const RState& s, const RDesc& d) {
    if constexpr (sizeof(V) == 8) {
        // integer cell values of magnitude <= 2^20: sums of up to four of
        // them, scaled by 2, 4 or 3 h (h a power of two), stay below 2^24
        auto small_int = [](double a) { return a == floor(a) && fabs(a) <= 1048576.0; };
        if (!c.cs.coef && small_int(d.a_incl) && small_int(d.a_matrix))
            refine_tile_dw<SCHEME, true>(c, tile, b, s, d);
        else
            refine_tile_dw<SCHEME, false>(c, tile, b, s, d);
    } else
        refine_tile_fp64<SCHEME>(c, tile, b, s, d);
}

// ITER step: inverse row Hartley of t on the tile + halo rows (z),
// p_new = z + beta p_old, x += alpha p_old (own rows), q = A p_new, p.q.
template <typename V, int SCHEME, int LOG2N>
__device__ __forceinline__ void fused_S_body(const Ctx& c, int tile, int b, const RState& s,
                                             const RDesc& d, double* red,
                                             typename ScalarOf<V>::T* bsc, unsigned* fxs,
                                             double* rowtab) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Sz<LOG2N> z(d.log2n);
    const int n = z.n;
    const int r0 = (tile - c.startS[b]) * d.tS;
    const int TR = min(d.tS, n - r0);   // own rows (the last tile may be shorter)
    const V* Pold = static_cast<const V*>(s.parity ? c.P1 : c.P0);
    V* Pnew = static_cast<V*>(s.parity ? c.P0 : c.P1);
    V* X = static_cast<V*>(c.X);
    V* Q = static_cast<V*>(c.Q);
    typedef typename ScalarOf<V>::T T;

    // ---- ITER ----
    // p_old (own and halo rows) and x (own rows) are read only after the
    // rows' transforms, t group by group: one thread per row asks for them
    // in L2 now, so those loads and copies wait on L2 instead of DRAM
    {
        const unsigned rb = (unsigned)(n * sizeof(V));
        const int k = threadIdx.x;
        if (k < TR + 2) prefetch_l2(Pold + node_at(d, z, (r0 - 1 + k) & (n - 1), 0), rb);
        else if (k >= 64 && k < 64 + TR) prefetch_l2(X + node_at(d, z, r0 + k - 64, 0), rb);
        else if (k >= 128 && k < 128 + TR + 2)
            prefetch_l2(static_cast<const V*>(c.T) + node_at(d, z, (r0 - 1 + k - 128) & (n - 1), 0), rb);
    }
    if (sizeof(V) == 16 && !c.cs.coef) fill_row_table<SCHEME>(rowtab, d.a_matrix, d.a_incl);
    // scalars of this step, converted once (thread 0) to the vector type
    if (threadIdx.x == 0) {
        bsc[0] = (T)s.beta[0];
        bsc[1] = (T)s.beta[1];
        bsc[2] = (T)s.alpha[0];
        bsc[3] = (T)s.alpha[1];
        bsc[4] = (T)d.a_incl;
        bsc[5] = (T)d.a_matrix;
    }
    const int SEQ = seq_stride(n);
    V* Pt = reinterpret_cast<V*>(smem_raw);            // (TR+2) padded rows
    // a tile of the whole realization: its halo rows are its own last and
    // first row, stored twice instead of transformed twice
    const bool whole = LOG2N <= 6 && TR == n;
    const int s0 = whole ? 1 : 0, slots = whole ? TR : TR + 2;   // slots to transform
    uint32_t* mrows = reinterpret_cast<uint32_t*>(Pt + (TR + 2) * SEQ);
    const int wpr = n >> 5;
    if (!c.cs.coef) {
        for (int w = threadIdx.x; w < (TR + 1) * wpr; w += blockDim.x) {
            const int mr = w / wpr, col = w - mr * wpr;
            const int row = (r0 - 1 + mr) & (n - 1);
            mrows[w] = __ldg(c.cs.mask + d.word_off + (((int64_t)row << z.log2n) >> 5) + col);
        }
    }
    __syncthreads();
    const TileCoef<T> tc{c.cs.coef ? nullptr : mrows, wpr, bsc[4], bsc[5]};
    const RowLayout<LOG2N> L(z.log2n);
    const T bx = bsc[0], by = bsc[1];
    const T alx = bsc[2], aly = bsc[3];
    const V* Tin = static_cast<const V*>(c.T);
    const V* tw = twiddles<V>(c.tb, n);
    // t of the rows of a transform group goes straight into the rows' own
    // shared slots by asynchronous copies (no registers held), one group
    // ahead: the copies of group g+1 are in flight while group g transforms
    // and while the stencil runs on the rows group g completed
    auto prefetch = [&](int g0) {
        const int q = s0 + g0 + L.qq;
        if (g0 + L.qq < slots) {
            const int row = (r0 - 1 + q) & (n - 1);
            V* buf = Pt + q * SEQ;
#pragma unroll
            for (int m = 0; m < 8; ++m)
                cp_async_v(buf + pidx(L.t + m * L.z.T), Tin + node_at(d, z, row, L.t + m * L.z.T));
        }
        cp_async_commit();   // an empty group past the last: uniform counting
    };
    prefetch(0);
    // q = A p on the own rows, once every row of the tile is transformed:
    // each thread walks down a column keeping the 3 x 3 neighbourhood (and
    // the two cell columns) in registers, so a node costs three shared loads
    // and two cell lookups.
    DotAcc<T> ax, ay;   // p.q
    // a thread walks down two columns j and j + 256 at once (n >= 512, the
    // kernel runs 256 threads): two independent chains of shared loads and
    // multiply-adds per row
    struct Win {
        V u0, u1, u2, m0, m1, m2;
        T cmm, cm0;
        int j, pm, p0, pp;
    };
    auto win_start = [&](Win& w, int j, int q0) {   // in front of own slot q0
        w.j = j;
        const int jm = (j - 1) & (n - 1), jp = (j + 1) & (n - 1);
        w.pm = pidx(jm); w.p0 = pidx(j); w.pp = pidx(jp);
        const V* up = Pt + (q0 - 1) * SEQ;
        const V* md = up + SEQ;
        w.u0 = up[w.pm]; w.u1 = up[w.p0]; w.u2 = up[w.pp];
        w.m0 = md[w.pm]; w.m1 = md[w.p0]; w.m2 = md[w.pp];
        w.cmm = tc.cell(c.cs, d, q0 - 1, r0 + q0 - 2, jm);
        w.cm0 = tc.cell(c.cs, d, q0 - 1, r0 + q0 - 2, j);
    };
    auto win_step = [&](Win& w, int q) {   // own slot q: node row r0 + q - 1
        const V* dn = Pt + (q + 1) * SEQ;
        const V d0 = dn[w.pm], d1 = dn[w.p0], d2 = dn[w.pp];
        const int jm = (w.j - 1) & (n - 1);
        const T c0m = tc.cell(c.cs, d, q, r0 + q - 1, jm);
        const T c00 = tc.cell(c.cs, d, q, r0 + q - 1, w.j);
        CellsT<T> a;
        a.mm = w.cmm;
        a.m0 = w.cm0;
        a.z0m = c0m;
        a.z00 = c00;
        const V qv = stencil_apply<SCHEME, V>(a, w.u0, w.u1, w.u2, w.m0, w.m1, w.m2, d0, d1, d2);
        Q[node_at(d, z, r0 + q - 1, w.j)] = qv;
        ax.add(w.m1.x, qv.x);
        ay.add(w.m1.y, qv.y);
        w.u0 = w.m0; w.u1 = w.m1; w.u2 = w.m2;
        w.m0 = d0; w.m1 = d1; w.m2 = d2;
        w.cmm = c0m; w.cm0 = c00;
    };
    // FP64: rows q0 .. q1 of column j by the weights (StencilRow)
    auto column64 = [&](int j, int q0, int q1) {
        if constexpr (sizeof(V) == 16) {
        const int jm = (j - 1) & (n - 1), jp = (j + 1) & (n - 1);
        const int pm = pidx(jm), p0 = pidx(j), pp = pidx(jp);
        const V* up = Pt + (q0 - 1) * SEQ;
        const V* md = up + SEQ;
        V u0 = up[pm], u1 = up[p0], u2 = up[pp], m0 = md[pm], m1 = md[p0], m2 = md[pp];
        // stored scaled by K (row_scale): alpha takes it out (finish_S)
        auto row = [&](const StencilRow& w, int q, auto doubled) {
            const V* dn = Pt + (q + 1) * SEQ;
            const V d0 = dn[pm], d1 = dn[p0], d2 = dn[pp];
            const V qv = apply_row<SCHEME, decltype(doubled)::value>(w, u0, u1, u2, m0, m1, m2, d0, d1, d2);
            Q[node_at(d, z, r0 + q - 1, j)] = qv;
            ax.add(m1.x, qv.x);
            ay.add(m1.y, qv.y);
            u0 = m0; u1 = m1; u2 = m2;
            m0 = d0; m1 = d1; m2 = d2;
        };
        if (tc.mrows) {
            auto bits = [&](int mrow) -> unsigned {   // cells (.., j-1), (.., j)
                const uint32_t* r = mrows + mrow * wpr;
                return ((r[jm >> 5] >> (jm & 31)) & 1u) | (((r[j >> 5] >> (j & 31)) & 1u) << 1);
            };
            unsigned top = bits(q0 - 1);
            for (int q = q0; q <= q1; ++q) {
                const unsigned bot = bits(q);
                row(table_row<SCHEME>(rowtab, top | (bot << 2)), q, std::true_type());
                top = bot;
            }
        } else {
            RowWalk<SCHEME> walk(tc.cell(c.cs, d, 0, r0 + q0 - 2, jm), tc.cell(c.cs, d, 0, r0 + q0 - 2, j));
            for (int q = q0; q <= q1; ++q)
                row(walk.step(tc.cell(c.cs, d, 0, r0 + q - 1, jm), tc.cell(c.cs, d, 0, r0 + q - 1, j)), q,
                    std::false_type());
        }
        }
    };
    // n < 256: 256 / n groups of threads share the tile's rows (at n = 64 the
    // columns alone kept 64 of 256 threads busy)
    auto stencil_rows = [&]() {
        constexpr bool TWO = sizeof(V) == 8 && LOG2N >= 9;   // n >= 512 = 2 x 256 threads
        constexpr int W = LOG2N < 8 ? 1 << LOG2N : 256;
        int q0 = 1, q1 = TR;
        if (W < 256) {
            const int per = (TR + 256 / W - 1) / (256 / W);
            q0 = 1 + (threadIdx.x / W) * per;
            q1 = min(TR, q0 + per - 1);
            if (q0 > q1) return;
        }
        for (int j = threadIdx.x & (W - 1); j < n; j += TWO ? 512 : 256) {
            if constexpr (sizeof(V) == 16) {
                column64(j, q0, q1);
                continue;
            }
            Win wa, wb;
            win_start(wa, j, q0);
            if (TWO) win_start(wb, j + 256, q0);
            for (int q = q0; q <= q1; ++q) {
                win_step(wa, q);
                if (TWO) win_step(wb, q);
            }
        }
    };
    // every row's transform is done by its own team of n/8 threads: the
    // barriers of the group loop are the team's, so the teams of a block
    // drift independently (one waits on its loads while another transforms)
    const TeamBar team(L.qq, L.z.T);
    for (int g0 = 0; g0 < slots; g0 += L.G) {
        const int q = s0 + g0 + L.qq;
        const bool active = g0 + L.qq < slots;
        const int row = (r0 - 1 + q) & (n - 1);
        const bool own = active && q >= 1 && q <= TR;
        prefetch(g0 + L.G);
        cp_async_wait<1>();   // this thread's copies of slot q have landed
        team();               // ... and those of the whole team
        V* buf = Pt + (active ? q : 0) * SEQ;
        V v[8];
        if (active) {
#pragma unroll
            for (int m = 0; m < 8; ++m) v[m] = buf[pidx(L.t + m * L.z.T)];
        }
        V pn[8];
        if constexpr (sizeof(V) == 16) hartley_row<LOG2N>(v, buf, L.t, tw, fx_twiddles(c.tb, n), active, fxs, team);
        else fft_reg<FFT_TO_BOTH, LOG2N>(v, buf, z.log2n, L.t, tw, active, team);
        if (active) {
            // p_new = z + beta p_old; own rows: x += alpha p_old (the lagged
            // solution update) and p_new out.  In two halves of four, the
            // global loads of a half before its stores (the compiler cannot
            // prove Pold, Pnew and X distinct)
#pragma unroll
            for (int h = 0; h < 8; h += 4) {
                V po[4], xo[4];
#pragma unroll
                for (int m = 0; m < 4; ++m) po[m] = Pold[node_at(d, z, row, L.t + (h + m) * L.z.T)];
                if (own) {
#pragma unroll
                    for (int m = 0; m < 4; ++m) xo[m] = X[node_at(d, z, row, L.t + (h + m) * L.z.T)];
                }
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const int k = L.t + (h + m) * L.z.T;
                    V zz = v[h + m];   // FP64: transformed by hartley_row
                    if constexpr (sizeof(V) == 8) zz = hartley_pair(zz, buf[pidx((n - k) & (n - 1))]);
                    pn[h + m] = axpy2(zz, bx, by, po[m]);
                }
                if (own) {
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        const int64_t node = node_at(d, z, row, L.t + (h + m) * L.z.T);
                        Pnew[node] = pn[h + m];
                        X[node] = axpy2(xo[m], alx, aly, po[m]);
                    }
                }
            }
        }
        team();   // the team's mirror reads of this row are done
        if (active) {
#pragma unroll
            for (int m = 0; m < 8; ++m) buf[pidx(L.t + m * L.z.T)] = pn[m];
            if (whole && (q == 1 || q == TR)) {
                V* twin = Pt + (q == 1 ? TR + 1 : 0) * SEQ;
#pragma unroll
                for (int m = 0; m < 8; ++m) twin[pidx(L.t + m * L.z.T)] = pn[m];
            }
        }
    }
    cp_async_wait<0>();
    __syncthreads();   // p_new of the whole tile visible
    stencil_rows();
    double sx = 0.0, sy = 0.0;
    block_sum2(ax, ay, red, sx, sy);
    if (threadIdx.x == 0) {
        c.partS[2 * (int64_t)tile] = sx;
        c.partS[2 * (int64_t)tile + 1] = sy;
    }
    finish_S(c, b, s, false, sizeof(V) == 16 ? row_scale<SCHEME>() : 1.0);
}

// The stencil pass of large grids (n >= 2^SPLIT_LOG2N, fused path) in two
// launches.  A tile of whole rows holds few of them there (4 to 6), and the two
// halo rows made their transforms 1.3 to 1.5 times the work at two blocks per
// SM.  Instead the row half transforms and updates every row once and stores p,
// and the stencil half (fused_Q_tile) reads p with its halo rows from L2: 56
// bytes per node pair instead of 48, no halo transforms, five blocks per SM.
// Per step: 2 x 2048^2 FP32 178 -> 142 us, 1024^2 FP64 130 -> 115 us.
constexpr int SPLIT_LOG2N = 10;
template <typename V, int LOG2N>
__device__ __forceinline__ void fused_P_body(const Ctx& c, int tile, int b, const RState& s,
                                             const RDesc& d, typename ScalarOf<V>::T* bsc,
                                             unsigned* fxs) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typedef typename ScalarOf<V>::T T;
    const RowLayout<LOG2N> L(d.log2n);
    const Sz<LOG2N>& z = L.z;
    const int n = z.n;
    const int r0 = (tile - c.startS[b]) * d.tS;
    const int TR = min(d.tS, n - r0);
    const int ng = (TR + L.G - 1) / L.G;
    const V* Pold = static_cast<const V*>(s.parity ? c.P1 : c.P0);
    V* Pnew = static_cast<V*>(s.parity ? c.P0 : c.P1);
    V* X = static_cast<V*>(c.X);
    const V* Tin = static_cast<const V*>(c.T);
    {   // rows read after their transforms: asked for in L2 now
        const unsigned rb = (unsigned)(n * sizeof(V));
        const int k = threadIdx.x;
        if (k < TR) prefetch_l2(Pold + node_at(d, z, r0 + k, 0), rb);
        else if (k >= 64 && k < 64 + TR) prefetch_l2(X + node_at(d, z, r0 + k - 64, 0), rb);
    }
    if (threadIdx.x == 0) {
        bsc[0] = (T)s.beta[0];
        bsc[1] = (T)s.beta[1];
        bsc[2] = (T)s.alpha[0];
        bsc[3] = (T)s.alpha[1];
    }
    const int SEQ = seq_stride(n);
    V* bufs = reinterpret_cast<V*>(smem_raw);   // two sets of L.G row buffers
    auto prefetch = [&](int g) {   // zhat of group g into row buffer set g & 1
        const int q = g * L.G + L.qq;
        if (g < ng && q < TR) {
            V* buf = bufs + ((g & 1) * L.G + L.qq) * SEQ;
#pragma unroll
            for (int m = 0; m < 8; ++m)
                cp_async_v(buf + pidx(L.t + m * z.T), Tin + node_at(d, z, r0 + q, L.t + m * z.T));
        }
        cp_async_commit();
    };
    prefetch(0);
    __syncthreads();
    const T bx = bsc[0], by = bsc[1], alx = bsc[2], aly = bsc[3];
    const V* tw = twiddles<V>(c.tb, n);
    const FxTw fx = fx_twiddles(c.tb, n);
    const TeamBar team(L.qq, z.T);
    for (int g = 0; g < ng; ++g) {
        const int q = g * L.G + L.qq;
        const bool active = q < TR;
        const int row = r0 + q;
        prefetch(g + 1);   // free since the barrier at the end of group g - 1
        cp_async_wait<1>();
        team();
        V* buf = bufs + ((g & 1) * L.G + (active ? L.qq : 0)) * SEQ;
        V v[8];
        if (active) {
#pragma unroll
            for (int m = 0; m < 8; ++m) v[m] = buf[pidx(L.t + m * z.T)];
        }
        hartley_row<LOG2N>(v, buf, L.t, tw, fx, active, fxs, team);
        if (active) {
#pragma unroll
            for (int h = 0; h < 8; h += 4) {   // a half's loads before its stores
                V po[4], xo[4];
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const int64_t node = node_at(d, z, row, L.t + (h + m) * z.T);
                    po[m] = Pold[node];
                    xo[m] = X[node];
                }
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const int64_t node = node_at(d, z, row, L.t + (h + m) * z.T);
                    Pnew[node] = axpy2(v[h + m], bx, by, po[m]);
                    X[node] = axpy2(xo[m], alx, aly, po[m]);
                }
            }
        }
        team();   // mirror reads of this row buffer are done
    }
    cp_async_wait<0>();
}

// The stencil half: q = A p on the tile's rows (FP64: K q, see StencilRow), p.q.
// A thread walks down two columns (FP32) or one (FP64).
template <typename V, int SCHEME>
__device__ void fused_Q_tile(const Ctx& c, int tile) {
    typedef typename ScalarOf<V>::T T;
    __shared__ double red[64];
    __shared__ T bsc[2];
    __shared__ __align__(16) double rowtab[sizeof(V) == 16 ? ROW_TABLE : 2];
    const int b = find_real(c.startS, c.batch, tile);
    const RState& s = c.st[b];
    if (s.phase != PH_ITER) return;
    const RDesc d = c.desc[b];
    if (d.log2n < SPLIT_LOG2N) return;
    const int n = d.n, m = n - 1, lg = d.log2n;
    const int r0 = (tile - c.startS[b]) * d.tS, r1 = min(r0 + d.tS, n);
    const V* __restrict__ P = static_cast<const V*>(s.parity ? c.P0 : c.P1) + d.node_off;
    V* __restrict__ Q = static_cast<V*>(c.Q) + d.node_off;
    const uint32_t* __restrict__ mw = c.cs.coef ? nullptr : c.cs.mask + d.word_off;
    const double* __restrict__ cf = c.cs.coef ? c.cs.coef + d.node_off : nullptr;
    if (sizeof(V) == 16) {
        if (mw) fill_row_table<SCHEME>(rowtab, d.a_matrix, d.a_incl);
    } else if (threadIdx.x == 0) {
        bsc[0] = (T)d.a_incl;
        bsc[1] = (T)d.a_matrix;
    }
    __syncthreads();
    DotAcc<T> ax, ay;
    auto word = [&](int i, int jj) { return __ldg(mw + ((((int64_t)(i & m)) << lg) + jj >> 5)) >> (jj & 31); };
    if constexpr (sizeof(V) == 16) {
        for (int j = threadIdx.x; j < n; j += blockDim.x) {
            const int jm = (j - 1) & m, jp = (j + 1) & m;
            auto at = [&](int i, int jj) { return __ldg(P + ((int64_t)(i & m) << lg) + jj); };
            V u0 = at(r0 - 1, jm), u1 = at(r0 - 1, j), u2 = at(r0 - 1, jp);
            V m0 = at(r0, jm), m1 = at(r0, j), m2 = at(r0, jp);
            auto row = [&](const StencilRow& w, int i, const V& d0, const V& d1, const V& d2, auto doubled) {
                const V q = apply_row<SCHEME, decltype(doubled)::value>(w, u0, u1, u2, m0, m1, m2, d0, d1, d2);
                Q[((int64_t)i << lg) + j] = q;
                ax.add(m1.x, q.x);
                ay.add(m1.y, q.y);
                u0 = m0; u1 = m1; u2 = m2;
                m0 = d0; m1 = d1; m2 = d2;
            };
            if (mw) {
                auto bits = [&](int i) -> unsigned { return (word(i, jm) & 1u) | ((word(i, j) & 1u) << 1); };
                unsigned top = bits(r0 - 1);
                for (int i = r0; i < r1; ++i) {
                    const V d0 = at(i + 1, jm), d1 = at(i + 1, j), d2 = at(i + 1, jp);
                    const unsigned bot = bits(i);
                    row(table_row<SCHEME>(rowtab, top | (bot << 2)), i, d0, d1, d2, std::true_type());
                    top = bot;
                }
            } else {
                auto cell = [&](int i, int jj) { return __ldg(cf + ((int64_t)(i & m) << lg) + jj); };
                RowWalk<SCHEME> walk(cell(r0 - 1, jm), cell(r0 - 1, j));
                for (int i = r0; i < r1; ++i) {
                    const V d0 = at(i + 1, jm), d1 = at(i + 1, j), d2 = at(i + 1, jp);
                    row(walk.step(cell(i, jm), cell(i, j)), i, d0, d1, d2, std::false_type());
                }
            }
        }
    } else {
        const float ai = bsc[0], am = bsc[1];
        struct Row { V l, a, b, r; };     // p at j - 1, j, j + 1, j + 2
        struct Cel { float l, a, b; };    // cells j - 1, j, j + 1
        for (int j = 2 * threadIdx.x; j < n; j += 2 * blockDim.x) {
            const int jm = (j - 1) & m, jp = (j + 2) & m;
            auto prow = [&](int i) -> Row {
                const V* p = P + ((int64_t)(i & m) << lg);
                const float4 v = __ldg(reinterpret_cast<const float4*>(p + j));
                return Row{__ldg(p + jm), make_float2(v.x, v.y), make_float2(v.z, v.w), __ldg(p + jp)};
            };
            auto crow = [&](int i) -> Cel {
                if (mw) {
                    const unsigned w = word(i, j), l = (j & 31) ? word(i, j - 1) : word(i, jm);
                    return Cel{(l & 1u) ? ai : am, (w & 1u) ? ai : am, (w & 2u) ? ai : am};
                }
                const double* p = cf + ((int64_t)(i & m) << lg);
                return Cel{(float)__ldg(p + jm), (float)__ldg(p + j), (float)__ldg(p + j + 1)};
            };
            Row u = prow(r0 - 1), v = prow(r0), ahead = prow(r0 + 1);
            Cel t = crow(r0 - 1), o = crow(r0);
#pragma unroll 2
            for (int i = r0; i < r1; ++i) {
                const Row dn = ahead;
                ahead = prow(i + 2);
                const Cel on = crow(i + 1);
                const V q0 = stencil_apply<SCHEME, V>(CellsT<float>{t.l, t.a, o.l, o.a}, u.l, u.a, u.b, v.l, v.a,
                                                      v.b, dn.l, dn.a, dn.b);
                const V q1 = stencil_apply<SCHEME, V>(CellsT<float>{t.a, t.b, o.a, o.b}, u.a, u.b, u.r, v.a, v.b,
                                                      v.r, dn.a, dn.b, dn.r);
                *reinterpret_cast<float4*>(Q + ((int64_t)i << lg) + j) = make_float4(q0.x, q0.y, q1.x, q1.y);
                ax.add(v.a.x, q0.x);
                ay.add(v.a.y, q0.y);
                ax.add(v.b.x, q1.x);
                ay.add(v.b.y, q1.y);
                u = v;
                v = dn;
                t = o;
                o = on;
            }
        }
    }
    double sx = 0.0, sy = 0.0;
    block_sum2(ax, ay, red, sx, sy);
    if (threadIdx.x == 0) {
        c.partS[2 * (int64_t)tile] = sx;
        c.partS[2 * (int64_t)tile + 1] = sy;
    }
    finish_S(c, b, s, false, sizeof(V) == 16 ? row_scale<SCHEME>() : 1.0);
}

// The refine or the stencil tile, by the realization's phase (`which`: 1
// refine, 2 stencil, 3 both: the profiler times the two apart).  SPLIT: the
// row half of the stencil on large grids.
enum { DO_REFINE = 1, DO_STENCIL = 2 };
template <typename V, int SCHEME, bool SPLIT>
__device__ void fused_RS_tile(const Ctx& c, int tile, int which) {
    __shared__ double red[64];   // block_sum2 scratch
    __shared__ unsigned fxs[8];  // row teams' reductions
    __shared__ typename ScalarOf<V>::T bsc[6];
    __shared__ __align__(16) double rowtab[sizeof(V) == 16 ? ROW_TABLE : 2];   // FP64: stencil rows
    const int b = find_real(c.startS, c.batch, tile);
    const RState& s = c.st[b];
    if (s.phase == PH_DONE || !(which & (s.phase == PH_REFINE ? DO_REFINE : DO_STENCIL))) return;
    const RDesc d = c.desc[b];
    if (s.phase == PH_REFINE) {
        refine_tile<V, SCHEME>(c, tile, b, s, d);
        return;
    }
    dispatch_size(d.log2n, [&]<int LG>() {
        if constexpr (SPLIT && LG >= SPLIT_LOG2N) fused_P_body<V, LG>(c, tile, b, s, d, bsc, fxs);
        else fused_S_body<V, SCHEME, LG>(c, tile, b, s, d, red, bsc, fxs, rowtab);
    });
}

// ----------------------------------------------------------- U kernel --
// The update kernel: tU rows per block, in transform groups of L.G rows
// (n/8 threads per row).  The residual is kept in the row-Hartley domain,
// rt = H r (H the unnormalised Hartley transform along rows, H H = n I):
// that is exactly what the column pass consumes, so the update writes it
// once instead of writing r and t = H r.
//   ITER    rt -= alpha H q  (H q by the row transform of q), |r|^2 = |rt|^2 / n;
//   REFINE  u = w (the new iterate), x = 0, r = r64 / |r64| (|r|^2 from r),
//           rt = H r.
// ITER streams: q of the next group arrives by asynchronous copies into the
// other of two row buffers while the current group transforms, and rt of a
// group is loaded before its transform.
template <typename V, int LOG2N>
__device__ __forceinline__ void fused_U_body(const Ctx& c, int blk, int b, const RState& s,
                                             const RDesc& d, double* red,
                                             typename ScalarOf<V>::T* usc, unsigned* fxs) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int phase = s.phase;
    const RowLayout<LOG2N> L(d.log2n);
    const Sz<LOG2N>& z = L.z;
    const int row0 = (blk - c.startU[b]) * d.tU;
    const int ng = (d.tU + L.G - 1) / L.G;   // transform groups of this block
    typedef typename ScalarOf<V>::T T;
    V* Rt = static_cast<V*>(c.R);
    V* X = static_cast<V*>(c.X);
    const V* Qv = static_cast<const V*>(c.Q);
    const int SEQ = seq_stride(z.n);
    V* bufs = reinterpret_cast<V*>(smem_raw);   // two sets of L.G row buffers
    const V* tw = twiddles<V>(c.tb, z.n);
    DotAcc<T> ax, ay;
    // each row by its own team of n/8 threads, which touches only its own row
    // buffers: team barriers only
    const TeamBar team(L.qq, z.T);
    const FxTw fx = fx_twiddles(c.tb, z.n);
    double inv_scale = 1.0;   // |r|^2 = (sum of the squares formed here) * inv_scale
    if (phase == PH_ITER) {
        // alpha = rho / p.q, formed by the last stencil block (finish_S)
        if (threadIdx.x == 0) {
            usc[0] = (T)c.uscal[4 * b];
            usc[1] = (T)c.uscal[4 * b + 1];
        }
        // rt of the block's rows is read group by group: one thread per row
        // asks for it in L2 now
        if (threadIdx.x < d.tU)
            prefetch_l2(Rt + node_at(d, z, row0 + threadIdx.x, 0), (unsigned)(z.n * sizeof(V)));
        auto prefetch = [&](int g) {   // q of group g into row buffer set g & 1
            const int q = g * L.G + L.qq;
            if (g < ng && q < d.tU) {
                V* buf = bufs + ((g & 1) * L.G + L.qq) * SEQ;
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    cp_async_v(buf + pidx(L.t + m * z.T), Qv + node_at(d, z, row0 + q, L.t + m * z.T));
            }
            cp_async_commit();
        };
        prefetch(0);
        __syncthreads();
        const T alx = usc[0], aly = usc[1];
        for (int g = 0; g < ng; ++g) {
            const int q = g * L.G + L.qq;
            const bool active = q < d.tU;
            const int row = row0 + q;
            // the other buffer set was last read by group g-1: the barrier at
            // the end of every group makes it free for group g+1's copies
            prefetch(g + 1);
            V rt[8];
            if (active && sizeof(V) == 8) {   // FP64: after the transform (registers)
#pragma unroll
                for (int m = 0; m < 8; ++m) rt[m] = Rt[node_at(d, z, row, L.t + m * z.T)];
            }
            cp_async_wait<1>();
            team();
            V* buf = bufs + ((g & 1) * L.G + (active ? L.qq : 0)) * SEQ;
            V v[8];
            if (active) {
#pragma unroll
                for (int m = 0; m < 8; ++m) v[m] = buf[pidx(L.t + m * z.T)];
            }
            hartley_row<LOG2N>(v, buf, L.t, tw, fx, active, fxs, team);
            if (active) {
                if (sizeof(V) == 16) {
#pragma unroll
                    for (int m = 0; m < 8; ++m) rt[m] = Rt[node_at(d, z, row, L.t + m * z.T)];
                }
#pragma unroll
                for (int m = 0; m < 8; ++m) {
                    const int k = L.t + m * z.T;
                    const V rr = axpy2(rt[m], -alx, -aly, v[m]);
                    Rt[node_at(d, z, row, k)] = rr;
                    ax.add(rr.x, rr.x);
                    ay.add(rr.y, rr.y);
                }
            }
            team();   // mirror reads of this row buffer are done
        }
        cp_async_wait<0>();
        inv_scale = 1.0 / (double)z.n;
    } else {
        float4* U4 = reinterpret_cast<float4*>(c.u);
        const V* Pold = static_cast<const V*>(s.parity ? c.P1 : c.P0);
        if constexpr (sizeof(T) == 4) {   // the same conversions as refine_tile_dw
            if (threadIdx.x == 0) {
                usc[0] = (float)s.s[0];
                usc[1] = (float)s.s[1];
                usc[2] = (float)s.alpha[0];
                usc[3] = (float)s.alpha[1];
                usc[4] = (float)c.uscal[4 * b];       // 1 / |r| per corrector (0 once
                usc[5] = (float)c.uscal[4 * b + 1];   // converged), from finish_S
            }
            __syncthreads();
        }
        for (int g = 0; g < ng; ++g) {
            const int q = g * L.G + L.qq;
            const bool active = q < d.tU;
            const int row = row0 + q;
            V* buf = bufs + (active ? L.qq : 0) * SEQ;
            V v[8];
            if constexpr (sizeof(T) == 4) {   // REFINE, mixed: u is a double word
                const DWScal k{usc[0], usc[1], usc[2], usc[3]};
                const float ix = usc[4], iy = usc[5];
                if (active) {
#pragma unroll
                    for (int h = 0; h < 8; h += 4) {
                        float4 uu[4];
                        V xx[4], pp[4], qv[4];
#pragma unroll
                        for (int m = 0; m < 4; ++m) {   // loads first, stores after
                            const int64_t node = node_at(d, z, row, L.t + (h + m) * z.T);
                            uu[m] = U4[node];
                            xx[m] = X[node];
                            pp[m] = Pold[node];
                            qv[m] = Qv[node];
                        }
#pragma unroll
                        for (int m = 0; m < 4; ++m) {
                            const int64_t node = node_at(d, z, row, L.t + (h + m) * z.T);
                            U4[node] = w_new(uu[m], xx[m], pp[m], k);
                            X[node] = mk<V>(0.f, 0.f);
                            const V rr = mk<V>(qv[m].x * ix, qv[m].y * iy);
                            v[h + m] = rr;
                            ax.add(rr.x, rr.x);
                            ay.add(rr.y, rr.y);
                        }
                    }
                }
            } else {   // REFINE, FP64
                // 1 / |r64| per corrector (0 once converged), from finish_S
                const double ix = c.uscal[4 * b], iy = c.uscal[4 * b + 1];
                if (active) {
#pragma unroll
                    for (int m = 0; m < 8; ++m) {
                        const int64_t node = node_at(d, z, row, L.t + m * z.T);
                        const double2 xx = to_d2(X[node]);
                        const double2 pp = to_d2(Pold[node]);
                        double2 uu = c.u[node];
                        uu.x += s.s[0] * (xx.x + s.alpha[0] * pp.x);
                        uu.y += s.s[1] * (xx.y + s.alpha[1] * pp.y);
                        c.u[node] = uu;
                        X[node] = from_d2<V>(make_double2(0.0, 0.0));
                        const double2 qq = to_d2(Qv[node]);
                        const V rr = from_d2<V>(make_double2(qq.x * ix, qq.y * iy));
                        v[m] = rr;
                        ax.add(rr.x, rr.x);
                        ay.add(rr.y, rr.y);
                    }
                }
            }
            hartley_row<LOG2N>(v, buf, L.t, tw, fx, active, fxs, team);
            if (active) {
#pragma unroll
                for (int m = 0; m < 8; ++m) Rt[node_at(d, z, row, L.t + m * z.T)] = v[m];
            }
            team();   // mirror reads of the buffer are done
        }
    }
    double sx = 0.0, sy = 0.0;
    block_sum2(ax, ay, red, sx, sy);
    if (threadIdx.x == 0) {
        c.partU[2 * (int64_t)blk] = sx * inv_scale;
        c.partU[2 * (int64_t)blk + 1] = sy * inv_scale;
    }
}

template <typename V>
__device__ void fused_U_tile(const Ctx& c, int blk) {
    __shared__ double red[64];   // block_sum2 scratch: 4 floats per warp (<= 32 warps)
    __shared__ typename ScalarOf<V>::T usc[6];
    __shared__ unsigned fxs[8];  // row teams' reductions
    const int b = find_real(c.startU, c.batch, blk);
    const RState& s = c.st[b];
    if (s.phase == PH_DONE) return;
    const RDesc d = c.desc[b];
    dispatch_size(d.log2n, [&]<int LG>() { fused_U_body<V, LG>(c, blk, b, s, d, red, usc, fxs); });
}

// ----------------------------------------------------------- C kernel --
// (the column solve body is in rve_colsolve.cuh)
// Column pass of one tile (any size): dispatches to the sized body.
// Reads the row transform of the residual (rt) from `in` and writes zhat to
// `out` (in == out allowed: every load of a column segment precedes its
// stores).
template <typename V>
__device__ void col_transform_tile(const V* in, V* out, const RDesc& d,
                                   int c0, V* smem, const Tables& tb, double delta, double* red,
                                   double* rho_part) {
    __shared__ typename ScalarOf<V>::T csc[1];
    dispatch_size(d.log2n, [&]<int LG>() {
        const Sz<LG> z(LG);
        col_solve_body<V, LG>([&](int r, int k) { return in[node_at(d, z, r, k)]; },
                              [&](int r, int k, V val) { out[node_at(d, z, r, k)] = val; }, d,
                              c0, smem, tb, delta, red, rho_part, csc);
    });
}

// `start`: of the tiles of this launch (c.startC, or those of a ColClass).
template <typename V>
__device__ void fused_C_tile(const Ctx& c, const int32_t* __restrict__ start, int blk) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[64];   // block_sum2 scratch: 4 floats per warp (<= 32 warps)
    const int b = find_real(start, c.batch, blk);
    if (c.st[b].phase == PH_DONE) return;
    const RDesc d = c.desc[b];
    const int tile = blk - start[b];
    col_transform_tile<V>(static_cast<const V*>(c.R), static_cast<V*>(c.T), d, tile * d.tC,
                          reinterpret_cast<V*>(smem_raw), c.tb, c.delta, red,
                          c.partC + 2 * (int64_t)(c.startC[b] + tile));
}

// ------------------------------------------------------ control kernel --
__device__ __forceinline__ bool bad(double v) { return !isfinite(v); }

// Stagnation test of an inner cycle: the residual must fall below
// STALL_FACTOR times its best value within STALL_STEPS steps.  Healthy
// preconditioned CG here contracts by ~0.8 per step or better, so only a
// cycle that has reached the attainable accuracy of its precision trips it.
constexpr double STALL_FACTOR = 0.7;
constexpr int STALL_STEPS = 30;

// Control step of realization b by one whole warp: lane k < 2 handles
// corrector k, with pU, pC its sums of the update and column passes.  (FP64
// square roots and divisions take about a microsecond each here: side by side
// for the two correctors, and alpha is the one finish_S formed.)
inline __device__ void control_apply(const Ctx& c, int b, double pU, double pC) {
    RState& s = c.st[b];
    const int k = threadIdx.x & 31;
    const bool mine = k < 2;
    const unsigned upto = k < 2 ? (2u << k) - 1u : 0u;   // correctors 0 .. k
    if (s.phase == PH_ITER) {
        const bool act = mine && s.active[k];
        const double alpha = act ? c.uscal[4 * b + 2 + k] : 0.0;
        const double rn = act ? sqrt(pU) : 0.0;
        const unsigned nan = __ballot_sync(0xffffffffu, act && (bad(alpha) || bad(rn) || bad(pC)));
        bool go = false, last = false;
        if (mine && !act) {
            if (!(nan & upto)) { s.alpha[k] = 0.0; s.beta[k] = 0.0; }
        } else if (act && !(nan & upto)) {
            s.alpha[k] = alpha;
            const int it = s.iters[k] + 1;
            s.iters[k] = it;
            // a cycle whose residual has stopped falling (the attainable
            // accuracy of the inner precision) ends early: the refinement
            // step then restarts from the true residual
            bool stalled = false;
            if (rn < STALL_FACTOR * s.best[k]) {
                s.best[k] = rn;
                s.stall[k] = 0;
            } else {
                const int st = s.stall[k] + 1;
                s.stall[k] = st;
                stalled = st >= STALL_STEPS;
            }
            if (rn <= s.target[k] || stalled || it >= c.max_iter) {
                s.active[k] = 0;       // frozen; alpha still pending for x
                s.beta[k] = 0.0;
                last = it >= c.max_iter && rn > s.target[k];
            } else {
                s.beta[k] = pC / s.rho[k];
                s.rho[k] = pC;
                go = true;
            }
        }
        const unsigned any = __ballot_sync(0xffffffffu, go), fin = __ballot_sync(0xffffffffu, last);
        if (k != 0) return;
        s.steps += 1;
        if (fin) s.final_pass = 1;
        if (nan) {
            s.status = RVE_ENAN;
            s.phase = PH_DONE;
            atomicAdd(c.ndone, 1);
            return;
        }
        s.parity ^= 1;
        if (!any) s.phase = PH_REFINE;   // every corrector ended its cycle
        return;
    }
    // REFINE: true residual of the accumulated solution
    const int refs = s.refinements + 1;
    const double rn = mine ? sqrt(c.uscal[4 * b + 2 + k]) : 0.0;
    const unsigned nan = __ballot_sync(0xffffffffu, mine && bad(rn));
    bool open = false, last = false;
    if (mine && !(nan & upto)) {
        if (refs == 1) s.fnorm[k] = rn;
        const double fn = s.fnorm[k];
        const bool conv = (refs == 1) ? (rn == 0.0) : (rn <= c.tol * fn);
        const double prev = s.relres[k];
        const double rel = fn > 0.0 ? rn / fn : 0.0;
        s.relres[k] = rel;
        s.alpha[k] = 0.0;
        // each cycle restarts CG from the true residual (p = z): keeping
        // the old direction across the replaced residual loses conjugacy
        // when the FP32 recurrence has drifted (tens of percent here)
        s.beta[k] = 0.0;
        if (conv || s.cdone[k]) {
            s.cdone[k] = 1;
            s.active[k] = 0;
            s.s[k] = 0.0;
        } else {
            open = true;
            s.s[k] = rn;
            s.active[k] = 1;
            s.best[k] = 1.0;   // the inner system starts from r / |r|
            s.stall[k] = 0;
            // inner target: what the outer tolerance still needs, but no less
            // than the usual inner reduction
            const double want = 0.5 * c.tol * fn / rn;
            double tgt = fmax(want, c.inner_tol);
            // a cycle gains at most what the rounding of its iterate allows
            // (about eps_inner times the condition of A on the correction): when
            // the last cycle's true residual fell far less than it was asked
            // to, ask the next one for no more than ten times what it achieved
            if (refs >= 2 && prev > 0.0) {
                const double got = rel / prev;
                if (got > 10.0 * s.target[k]) tgt = fmax(tgt, 0.1 * got);
            }
            s.target[k] = fmin(0.5, tgt);
            s.rho[k] = pC;
            last = s.iters[k] >= c.max_iter;
        }
    }
    const unsigned any = __ballot_sync(0xffffffffu, open), fin = __ballot_sync(0xffffffffu, last);
    if (k != 0) return;
    s.refinements = refs;
    if (fin) s.final_pass = 1;
    if (nan) {
        s.status = RVE_ENAN;
        s.phase = PH_DONE;
        atomicAdd(c.ndone, 1);
        return;
    }
    if (!any || s.final_pass) {
        if (any) s.status = RVE_ENOCONV;
        s.phase = PH_DONE;
        atomicAdd(c.ndone, 1);
        return;
    }
    s.phase = PH_ITER;
}

// ------------------------------------------------------- launchers --
// Instantiated per vector type and scheme: the fused kernels in rve_pipe32.cu
// and rve_pipe64.cu, the persistent kernel in rve_persist32.cu and
// rve_persist64.cu (one unit each, so that they compile side by side).
// One pipeline step (with `ev`: PROFILE_KERNELS + 1 events around its launches).
template <typename V, int SCHEME>
cudaError_t fused_step(const Plan& p, const Ctx& c, cudaStream_t s, cudaEvent_t* ev);
template <typename V, int SCHEME> cudaError_t set_smem_attrs(const Plan& p);
template <typename V, int SCHEME> rve_status persistent_prepare_t(Plan& p);
template <typename V, int SCHEME>
rve_status persistent_launch(const Plan& p, const Ctx& c, const rve_solve_opts& o, cudaStream_t s);
cudaError_t launch_control(const Plan& p, const Ctx& c, cudaStream_t s);

}  // namespace rve
