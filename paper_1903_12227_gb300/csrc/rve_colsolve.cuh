// rve_colsolve.cuh -- the column pass of the preconditioner: periodic
// tridiagonal solves along one grid axis after the Hartley transforms along
// the others (shared by the 2D pipeline and the 3D solver).
#pragma once

#include "rve_common.cuh"

namespace rve {

// Column pass on t = row-Hartley(r).  The row transform diagonalises the
// row factor of A_Delta, so column k2 of t is left with the periodic
// tridiagonal system
//     M z = t,   M = c0 (T + lambda) + delta,   lambda = 4 sin^2(pi k2 / n),
// T the periodic second difference along the column (the fast Poisson
// scheme of Hockney: Fourier in one direction, tridiagonal solves in the
// other).  With rho + 1/rho = 2 + mu, mu = lambda + delta / c0,
//     M = (c0 / rho) (1 - rho S)(1 - rho S^T),   S the cyclic shift,
// so M^{-1} t = (rho / c0) F^T F t with the causal filter F = (1 - rho S)^{-1}
// (y_i = t_i + rho y_{i-1}, periodic) and its transpose, the anticausal
// filter.  The pass stores zhat = M^{-1} t / n (the row transform in the
// stencil kernel supplies the other factor 1/n of the inverse transform)
// and rho_c = r.z = t.zhat = (rho / (n c0)) |F t|^2.
//
// Each thread holds SEG consecutive rows of one column in registers: it
// runs the filter over its segment from a zero start, the segment's end
// value goes through shared memory, and every thread adds the periodic
// carry-in  sum_{j=1..P} R^{j-1} e_{s-j} / (1 - R^P)  (R = rho^SEG, P
// segments; the sum stops once R^{j-1} is negligible) times rho^{i+1}.
// The anticausal filter runs the same way upwards.
//
// FP64 columns of 16 or more segments take their carries from a warp scan
// (col_carries) instead: the sum over P segments in each of P threads was 64
// terms of 4 FP64 operations per 16 rows at n = 1024, against 12 per row for
// the filters.  There the segment is read twice from registers, once for its
// end value and once with the carry known, which saves the powers of rho
// (12 FP64 operations per row instead of 14).  1024^2, one realization: 230 us ->
// 51 us per pass; preconditioner column pass of 25 x 512^2: 342 -> 196 us.  The singular column
// k2 = 0 with delta = 0 (rho = 1) takes the pseudo-inverse: with
// t' = t - mean t, y = cumsum t' made mean-zero, w = reverse cumsum y made
// mean-zero, zhat = w / (n c0), rho_c = |y|^2 / (n c0).
// Block: C columns x P segments, thread (cc, s) with cc fastest so that the
// global accesses of a warp are row segments of C elements.  `rho_part`
// may be null.  rho_of(k2) gives the filter root of column k2 (not called
// for the singular column).  UNROLL: the periodic carries sum all P segment
// values (independent loads, no early exit) instead of stopping once the
// weight is negligible.  SEGO > 0 sets the rows per segment (a divisor of
// n) in place of col_seg_rows.

// Carries of one column's P segment values by W = min(P, 32) lanes of a warp,
// in place: X[s C] (the end of segment s, from a zero start) becomes the carry
// into segment s of the periodic recurrence c_{s+1} = X_s + R c_s (DOWN: run
// from the last segment to the first).  `singular` (R = 1): the running sums
// from zero, and the total to *tot.  Powers below 1e-19 end the scan.
struct ColScan {   // per lane, kept for the second filter
    double R, RK, inv;
};
template <int P, int SEG>
__device__ __forceinline__ ColScan col_scan_of(double rho, bool singular) {
    constexpr int W = P < 32 ? P : 32, K = P / W;
    ColScan q;
    q.R = rho;
#pragma unroll
    for (int k = 1; k < SEG; k <<= 1) q.R *= q.R;
    q.RK = q.R;
#pragma unroll
    for (int k = 1; k < K; k <<= 1) q.RK *= q.RK;
    double RP = q.RK;
#pragma unroll
    for (int k = 1; k < W; k <<= 1) RP = RP < 1e-19 ? 0.0 : RP * RP;
    q.inv = (singular || RP < 1e-19) ? 1.0 : 1.0 / (1.0 - RP);
    return q;
}
template <int P, bool DOWN>
__device__ __forceinline__ void col_carries(double2* X, int C, const ColScan& q, bool singular,
                                            double2* tot) {
    constexpr int W = P < 32 ? P : 32, K = P / W;
    const int l = threadIdx.x & (W - 1);
    auto at = [&](int k) -> double2& { const int s = l * K + k; return X[(DOWN ? P - 1 - s : s) * C]; };
    double2 e[K], a = make_double2(0.0, 0.0);
#pragma unroll
    for (int k = 0; k < K; ++k) {
        e[k] = at(k);
        a.x = fma(q.R, a.x, e[k].x);
        a.y = fma(q.R, a.y, e[k].y);
    }
    double f = q.RK, pw = 1.0;   // RK^d, RK^l
#pragma unroll
    for (int d = 1; d < W; d <<= 1) {
        if (__all_sync(0xffffffffu, f < 1e-19)) {   // terms that far off vanish
            if (l >= d) pw = 0.0;
            break;
        }
        const double x = __shfl_up_sync(0xffffffffu, a.x, d, W), y = __shfl_up_sync(0xffffffffu, a.y, d, W);
        if (l >= d) {
            a.x = fma(f, x, a.x);
            a.y = fma(f, y, a.y);
        }
        if (l & d) pw *= f;
        f *= f;
    }
    const double tx = __shfl_sync(0xffffffffu, a.x, W - 1, W), ty = __shfl_sync(0xffffffffu, a.y, W - 1, W);
    double cx = __shfl_up_sync(0xffffffffu, a.x, 1, W), cy = __shfl_up_sync(0xffffffffu, a.y, 1, W);
    if (l == 0) cx = cy = 0.0;
    if (singular) {
        if (l == 0) *tot = make_double2(tx, ty);
    } else {
        cx = fma(pw, tx * q.inv, cx);
        cy = fma(pw, ty * q.inv, cy);
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        at(k) = make_double2(cx, cy);
        cx = fma(q.R, cx, e[k].x);
        cy = fma(q.R, cy, e[k].y);
    }
}

// The FP64 column pass with scanned carries (see above); the singular
// column's arithmetic is that of col_solve_core.
template <int LOG2N, int SEG, typename Ld, typename St, typename RhoOf>
__device__ __forceinline__ void col_solve_scan(Ld&& ld, St&& st, RhoOf&& rho_of, const RDesc& d,
                                               int c0, double2* smem, double delta, double* red,
                                               double* rho_part, double* csc) {
    constexpr int n = 1 << LOG2N, P = n / SEG, W = P < 32 ? P : 32;
    const int C = d.tC, tid = threadIdx.x;
    const int s = tid / C, cc = tid - s * C;
    const bool active = s < P;
    const int k2 = c0 + cc;
    const bool zero_block = (c0 == 0 && delta == 0.0);   // block holds the singular column
    const bool zcol = zero_block && cc == 0;
    double2* E = smem;                                        // [P][C] segment values, then carries
    double2* Zs = smem + 2 * P * C;                           // [2][P] singular column: segment sums
    double* roots = reinterpret_cast<double*>(smem + P * C);  // [C]
    double2* tot = smem + P * C + C;                          // totals of the singular column
    double2 v[SEG];
#pragma unroll
    for (int i = 0; i < SEG; ++i) v[i] = active ? ld(s * SEG + i, k2) : make_double2(0.0, 0.0);
    if (s == 0) roots[cc] = zcol ? 1.0 : rho_of(k2);
    if (tid == 0) csc[0] = 1.0 / ((double)n * d.c0);
    __syncthreads();
    const double rho = roots[cc];
    // C P <= blockDim.x: a warp scans the columns of at most one group of lanes
    const int scol = tid / W;
    const bool scans = (tid >> 5) * (32 / W) < C;   // warp-uniform
    const bool szcol = zero_block && scol == 0;
    const int sc_ = scol < C ? scol : 0;
    {
        double2 e = v[0];
#pragma unroll
        for (int i = 1; i < SEG; ++i) {
            e.x = fma(rho, e.x, v[i].x);
            e.y = fma(rho, e.y, v[i].y);
        }
        if (active) E[s * C + cc] = e;
    }
    ColScan q{};
    if (scans) q = col_scan_of<P, SEG>(roots[sc_], szcol);
    __syncthreads();
    if (scans && scol < C) col_carries<P, false>(E + scol, C, q, szcol, tot);
    __syncthreads();
    const double inv_nc0 = csc[0];
    {
        const double2 c = active ? E[s * C + cc] : make_double2(0.0, 0.0);
        v[0].x = fma(rho, c.x, v[0].x);
        v[0].y = fma(rho, c.y, v[0].y);
#pragma unroll
        for (int i = 1; i < SEG; ++i) {
            v[i].x = fma(rho, v[i - 1].x, v[i].x);
            v[i].y = fma(rho, v[i - 1].y, v[i].y);
        }
    }
    double wbx = 0.0, wby = 0.0;   // singular column: mean of w
    if (zero_block) {              // block-uniform: y = cumsum(t - mean t), made mean-zero
        if (zcol && active) {
            const double mx = tot[0].x / (double)n, my = tot[0].y / (double)n;
            double2 s1 = make_double2(0.0, 0.0), s2 = s1;
#pragma unroll
            for (int i = 0; i < SEG; ++i) {
                const double k = (double)(s * SEG + i + 1);
                v[i].x -= k * mx;
                v[i].y -= k * my;
                s1.x += v[i].x;
                s1.y += v[i].y;
                s2.x += k * v[i].x;
                s2.y += k * v[i].y;
            }
            Zs[s] = s1;
            Zs[P + s] = s2;
        }
        __syncthreads();
        if (tid < 32) {   // sums over the segments
            double t[4] = {0.0, 0.0, 0.0, 0.0};
            for (int j = tid; j < P; j += 32) {
                t[0] += Zs[j].x;
                t[1] += Zs[j].y;
                t[2] += Zs[P + j].x;
                t[3] += Zs[P + j].y;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) t[k] = warp_sum(t[k]);
            if (tid == 0) {
                tot[0] = make_double2(t[0], t[1]);
                tot[1] = make_double2(t[2], t[3]);
            }
        }
        __syncthreads();
        if (zcol && active) {
            const double ybx = tot[0].x / (double)n, yby = tot[0].y / (double)n;
            const double tri = 0.5 * (double)(n + 1);   // (1/n) sum_{j=1..n} j
            wbx = tot[1].x / (double)n - ybx * tri;
            wby = tot[1].y / (double)n - yby * tri;
#pragma unroll
            for (int i = 0; i < SEG; ++i) { v[i].x -= ybx; v[i].y -= yby; }
        }
    }
    const double sc = rho * inv_nc0;
    // rho partials: (rho / (n c0)) |F t|^2 per corrector
    DotAcc<double> ax, ay;
    if (active) {
        double qx = 0.0, qy = 0.0;
#pragma unroll
        for (int i = 0; i < SEG; ++i) {
            qx = fma(v[i].x, v[i].x, qx);
            qy = fma(v[i].y, v[i].y, qy);
        }
        ax.add(sc, qx);
        ay.add(sc, qy);
    }
    {
        double2 e = v[SEG - 1];
#pragma unroll
        for (int i = SEG - 2; i >= 0; --i) {
            e.x = fma(rho, e.x, v[i].x);
            e.y = fma(rho, e.y, v[i].y);
        }
        if (active) E[s * C + cc] = e;   // only this thread read the carry there
    }
    __syncthreads();
    if (scans && scol < C) col_carries<P, true>(E + scol, C, q, szcol, tot + 2);
    __syncthreads();
    if (active) {
        const double2 c = E[s * C + cc];
        v[SEG - 1].x = fma(rho, c.x, v[SEG - 1].x);
        v[SEG - 1].y = fma(rho, c.y, v[SEG - 1].y);
#pragma unroll
        for (int i = SEG - 2; i >= 0; --i) {
            v[i].x = fma(rho, v[i + 1].x, v[i].x);
            v[i].y = fma(rho, v[i + 1].y, v[i].y);
        }
#pragma unroll
        for (int i = SEG - 1; i >= 0; --i)
            st(s * SEG + i, k2, zcol ? make_double2((v[i].x - wbx) * sc, (v[i].y - wby) * sc)
                                     : make_double2(v[i].x * sc, v[i].y * sc));
    }
    if (rho_part) {
        double sx = 0.0, sy = 0.0;
        block_sum2(ax, ay, red, sx, sy);
        if (tid == 0) { rho_part[0] = sx; rho_part[1] = sy; }
    }
}

template <typename V, int LOG2N, bool UNROLL = false, int SEGO = 0, typename Ld, typename St,
          typename RhoOf>
__device__ __forceinline__ void col_solve_core(Ld&& ld, St&& st, RhoOf&& rho_of, const RDesc& d,
                                               int c0, V* smem, const Tables& tb, double delta,
                                               double* red, double* rho_part,
                                               typename ScalarOf<V>::T* csc) {
    typedef typename ScalarOf<V>::T Ts;
    constexpr int n = 1 << LOG2N;
    constexpr int SEG = SEGO > 0 ? SEGO : col_seg_rows(n, (int)sizeof(V));
    constexpr int P = n / SEG;
    // carry terms below this weight are dropped (far below the rounding of Ts)
    constexpr Ts CARRY_EPS = sizeof(Ts) == 4 ? (Ts)1e-10 : (Ts)1e-19;
    const Sz<LOG2N> z(LOG2N);
    const int C = d.tC;
    const int tid = threadIdx.x;
    const int s = tid / C, cc = tid - (tid / C) * C;
    const bool active = s < P;
    const int k2 = c0 + cc;
    const bool zero_block = (c0 == 0 && delta == 0.0);   // block holds the singular column
    const bool zcol = zero_block && cc == 0;
    if (tid == 0) csc[0] = (Ts)(1.0 / ((double)n * d.c0));
    V v[SEG];
#pragma unroll
    for (int i = 0; i < SEG; ++i)
        v[i] = active ? ld(s * SEG + i, k2) : mk<V>((Ts)0, (Ts)0);
    Ts rho = (Ts)1;
    if (active && !zcol) rho = rho_of(k2);
    V* E = smem;                  // [P][C] segment end values (causal pass)
    V* B = smem + P * C;          // [P][C] segment start values (anticausal pass)
    V* Zs = smem + 2 * P * C;     // [2][P] singular column: segment sums
    // causal filter within the segment
#pragma unroll
    for (int i = 1; i < SEG; ++i) {
        v[i].x += rho * v[i - 1].x;
        v[i].y += rho * v[i - 1].y;
    }
    if (active) E[s * C + cc] = v[SEG - 1];
    __syncthreads();   // also publishes csc
    const Ts inv_nc0 = csc[0];
    Ts R = (Ts)0, inv1mRP = (Ts)0;
    if (active && !zcol) {
        R = rho;
#pragma unroll
        for (int k = 1; k < SEG; k <<= 1) R *= R;            // rho^SEG
        Ts RP = R;
#pragma unroll
        for (int k = 1; k < P; k <<= 1) RP *= RP;            // rho^n
        inv1mRP = (Ts)1 / ((Ts)1 - RP);
        V acc = mk<V>((Ts)0, (Ts)0);
        Ts Rj = (Ts)1;
        if (UNROLL) {
#pragma unroll
            for (int j = 1; j <= P; ++j) {
                const V e = E[((s - j) & (P - 1)) * C + cc];
                acc.x += Rj * e.x;
                acc.y += Rj * e.y;
                Rj *= R;
            }
        } else {
            for (int j = 1; j <= P; ++j) {
                const V e = E[((s - j) & (P - 1)) * C + cc];
                acc.x += Rj * e.x;
                acc.y += Rj * e.y;
                Rj *= R;
                if (Rj < CARRY_EPS) break;
            }
        }
        const Ts cx = acc.x * inv1mRP, cy = acc.y * inv1mRP;
        Ts pw = rho;
#pragma unroll
        for (int i = 0; i < SEG; ++i) {
            v[i].x += pw * cx;
            v[i].y += pw * cy;
            pw *= rho;
        }
    } else if (active) {   // singular column: y = cumsum(t - mean t)
        V tot = mk<V>((Ts)0, (Ts)0), pre = mk<V>((Ts)0, (Ts)0);
        for (int j = 0; j < P; ++j) {
            const V e = E[j * C];
            tot.x += e.x;
            tot.y += e.y;
            if (j < s) { pre.x += e.x; pre.y += e.y; }
        }
        const Ts mx = tot.x / (Ts)n, my = tot.y / (Ts)n;
#pragma unroll
        for (int i = 0; i < SEG; ++i) {
            const Ts k = (Ts)(s * SEG + i + 1);
            v[i].x += pre.x - k * mx;
            v[i].y += pre.y - k * my;
        }
    }
    Ts wbx = (Ts)0, wby = (Ts)0;   // singular column: mean of w
    if (zero_block) {              // block-uniform
        if (zcol && active) {
            V s1 = mk<V>((Ts)0, (Ts)0), s2 = mk<V>((Ts)0, (Ts)0);
#pragma unroll
            for (int i = 0; i < SEG; ++i) {
                const Ts k = (Ts)(s * SEG + i + 1);
                s1.x += v[i].x; s1.y += v[i].y;
                s2.x += k * v[i].x; s2.y += k * v[i].y;
            }
            Zs[s] = s1;
            Zs[P + s] = s2;
        }
        __syncthreads();
        if (zcol && active) {
            V t1 = mk<V>((Ts)0, (Ts)0), t2 = mk<V>((Ts)0, (Ts)0);
            for (int j = 0; j < P; ++j) {
                t1.x += Zs[j].x; t1.y += Zs[j].y;
                t2.x += Zs[P + j].x; t2.y += Zs[P + j].y;
            }
            const Ts ybx = t1.x / (Ts)n, yby = t1.y / (Ts)n;
            const Ts tri = (Ts)0.5 * (Ts)(n + 1);   // (1/n) sum_{j=1..n} j
            wbx = t2.x / (Ts)n - ybx * tri;
            wby = t2.y / (Ts)n - yby * tri;
#pragma unroll
            for (int i = 0; i < SEG; ++i) { v[i].x -= ybx; v[i].y -= yby; }
        }
    }
    // rho partials: (rho / (n c0)) |F t|^2 per corrector
    DotAcc<Ts> ax, ay;
    if (active) {
        Ts qx = (Ts)0, qy = (Ts)0;
#pragma unroll
        for (int i = 0; i < SEG; ++i) {
            qx += v[i].x * v[i].x;
            qy += v[i].y * v[i].y;
        }
        const Ts wgt = rho * inv_nc0;
        ax.add(wgt, qx);
        ay.add(wgt, qy);
    }
    // anticausal filter within the segment
#pragma unroll
    for (int i = SEG - 2; i >= 0; --i) {
        v[i].x += rho * v[i + 1].x;
        v[i].y += rho * v[i + 1].y;
    }
    if (active) B[s * C + cc] = v[0];
    __syncthreads();
    if (active) {
        Ts sc, wx, wy;
        if (!zcol) {
            V acc = mk<V>((Ts)0, (Ts)0);
            Ts Rj = (Ts)1;
            if (UNROLL) {
#pragma unroll
                for (int j = 1; j <= P; ++j) {
                    const V e = B[((s + j) & (P - 1)) * C + cc];
                    acc.x += Rj * e.x;
                    acc.y += Rj * e.y;
                    Rj *= R;
                }
            } else {
                for (int j = 1; j <= P; ++j) {
                    const V e = B[((s + j) & (P - 1)) * C + cc];
                    acc.x += Rj * e.x;
                    acc.y += Rj * e.y;
                    Rj *= R;
                    if (Rj < (Ts)1e-18) break;
                }
            }
            wx = acc.x * inv1mRP;
            wy = acc.y * inv1mRP;
            sc = rho * inv_nc0;
        } else {   // w = reverse cumsum of y, then mean-zero
            V suf = mk<V>((Ts)0, (Ts)0);
            for (int j = s + 1; j < P; ++j) { suf.x += B[j * C].x; suf.y += B[j * C].y; }
            wx = suf.x;
            wy = suf.y;
            sc = inv_nc0;
        }
        Ts pw = zcol ? (Ts)0 : rho;
#pragma unroll
        for (int i = SEG - 1; i >= 0; --i) {
            const Ts gx = zcol ? (wx - wbx) : pw * wx;
            const Ts gy = zcol ? (wy - wby) : pw * wy;
            st(s * SEG + i, k2, mk<V>((v[i].x + gx) * sc, (v[i].y + gy) * sc));
            pw *= rho;
        }
    }
    if (rho_part) {
        double sx = 0.0, sy = 0.0;
        block_sum2(ax, ay, red, sx, sy);
        if (tid == 0) { rho_part[0] = sx; rho_part[1] = sy; }
    }
}

// The column pass of the 2D pipeline: the root from the table (delta = 0)
// or, rarely, computed in FP64 for the shift delta.
template <typename V, int LOG2N, typename Ld, typename St>
__device__ __forceinline__ void col_solve_body(Ld&& ld, St&& st, const RDesc& d, int c0,
                                               V* smem, const Tables& tb, double delta,
                                               double* red, double* rho_part,
                                               typename ScalarOf<V>::T* csc) {
    typedef typename ScalarOf<V>::T Ts;
    constexpr int n = 1 << LOG2N;
    auto root = [&](int k2) -> Ts {
        return (delta == 0.0) ? rho_table<Ts>(tb, n)[k2]
                              : (Ts)filter_root(tb.lap[n + k2] + delta / d.c0);
    };
    if constexpr (sizeof(Ts) == 8)
        col_solve_scan<LOG2N, col_seg_rows(n, 16)>(ld, st, root, d, c0, smem, delta, red, rho_part, csc);
    else
        col_solve_core<V, LOG2N>(ld, st, root, d, c0, smem, tb, delta, red, rho_part, csc);
}

}  // namespace rve
