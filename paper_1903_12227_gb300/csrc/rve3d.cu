// rve3d.cu -- the 3D extension of the RVE corrector method (the setting of
// Sec. 2 carries over to d = 3; the rank-3 Kronecker Laplacian of Sec. 3.2
// and Eq. "As_Kron_d"; multilinear functions on cubes, Sec. 3.1): cubes on
// the torus [0,L)^3, the trilinear Q1 element K1(x)M1(x)M1 + M1(x)K1(x)M1 +
// M1(x)M1(x)K1, three corrector problems solved by PCG with B = c0 A_Delta +
// delta I (A_Delta the periodic 7-point Laplacian), and the 3x3 homogenized
// matrix.
//
// Grid: n = L m0 nodes per axis, node (i,j,k) at ((i n + j) n + k) within
// the realization; cell (i,j,k) has lower corner node (i,j,k); local corner
// a = 4 a1 + 2 a2 + a3.  The three correctors travel as two pairs: (u_1,
// u_2) and (u_3, 0), so that every kernel -- the stencil, the Hartley
// transforms (pair-packed complex FFT) and the column solve -- works on the
// pair layout of the 2D path.
//
// Units.  The solver's unit of work is one pair of one realization.  Units
// are numbered by grid size (within a size, the pair-0 units first), and
// every launch covers the consecutive units of one size, each unit with its
// own scalars and flags; a unit that has finished makes its blocks return
// at once.  The host polls the flags every few steps.
//
// Preconditioner: the Hartley transforms along x (contiguous lines) and y
// (lines of stride n) diagonalise two factors of A_Delta; along z (lines of
// stride n^2) each (kx, ky) leaves the periodic tridiagonal system
// c0 (T + lambda(kx) + lambda(ky)) + delta, solved by the causal/anticausal
// filter pair of the 2D column pass (rve_colsolve.cuh).  B^{-1} = n^-2 Hx
// Hy M^-1 Hy Hx.
//
// Precision.  GB300 runs FP64 at 1/64 of the FP32 rate, and the 3D stencil
// and transforms carry enough arithmetic per node to be bound by it.  Both
// paths run PCG cycles (Saad, Iterative Methods for Sparse Linear Systems,
// Algorithm 9.1) on A e = r64 / s from e = 0, s = |r64|, between FP64 true
// residuals r64 = f - A u (iterative refinement, u += s e), until |r64| <=
// tol |f|.  FP64: the cycle's vectors are FP64 and it runs to the outer
// tolerance, so one cycle is textbook PCG and a second one is rare.
// Mixed: the cycle's vectors and arithmetic are FP32 and it stops at a
// relative reduction max(tol |f| / (2 |r64|), inner_tol).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <type_traits>
#include <vector>

#include "rve_colsolve.cuh"
#include "rve_common.cuh"
#include "rve_internal.h"

namespace rve {

// Descriptor of one unit (a corrector pair of a realization).
struct U3 {
    int32_t n, log2n, pair, pad2;
    int32_t n_incl, s;
    int32_t real;       // realization index
    int32_t partner;    // the realization's other unit
    int64_t off;        // first node of the unit's vectors
    int64_t cell_off;   // first cell (= node) of the realization: mask, coef, ABI vectors
    int64_t part_off;   // first partial (doubles) of the unit
    double am, ai, h, c0, inv_vol;
    float am32, ai32;
    uint64_t key;       // SplitMix64 key of the realization
};

// Blocks of a launch over the units of one grid size (consecutive unit ids
// from `first`): block -> (unit, block within the unit).
struct Grp {
    const U3* __restrict__ desc;
    int first;          // first unit of the launch
    int per_log2;       // log2 of the blocks per unit
};
__device__ __forceinline__ int unit_of(const Grp& g, int& lb) {
    lb = blockIdx.x & ((1 << g.per_log2) - 1);
    return g.first + (blockIdx.x >> g.per_log2);
}

// Local index of node (i, j, k) (periodic) within a realization.
__device__ __forceinline__ int l3(const U3& d, int i, int j, int k) {
    const int m = d.n - 1;
    return ((((i & m) << d.log2n) + (j & m)) << d.log2n) + (k & m);
}

// Cell values in the arithmetic type T: a byte mask with the two values, or
// an explicit array.
template <typename T> struct Cells3T {
    const uint8_t* __restrict__ mask;
    const T* __restrict__ coef;
};
template <typename T> __device__ __forceinline__ T two_values(const U3& d, bool incl);
template <> __device__ __forceinline__ double two_values<double>(const U3& d, bool incl) { return incl ? d.ai : d.am; }
template <> __device__ __forceinline__ float two_values<float>(const U3& d, bool incl) { return incl ? d.ai32 : d.am32; }

constexpr int T3 = 256;   // threads of the node kernels
constexpr int SZ = 4;     // stencil: consecutive planes per thread
constexpr int Z_THREADS = 512;   // z solve

// Block sums of two per-thread values (x, y), valid in thread 0: an xor
// butterfly within each warp in the values' own precision, then the warp
// sums in FP64 in warp order (fixed order: deterministic).  A thread's
// value sums only its own few nodes, so an FP32 tree stays short.
// `red` holds 2 * (blockDim.x / 32) doubles.
template <typename T>
__device__ __forceinline__ void block_pair_sum(T x, T y, double* red, double& sx, double& sy) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        red[2 * wid] = (double)x;
        red[2 * wid + 1] = (double)y;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            a += red[2 * w];
            b += red[2 * w + 1];
        }
        sx = a;
        sy = b;
    }
}

// --------------------------------------------------------------- field --
// One thread per (cube, row d1, d2): sets the s cells along the third axis.
__global__ void k3_gen_field(const U3 d, uint8_t* __restrict__ mask) {
    const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t rows = (int64_t)d.n_incl * d.s * d.s;
    if (gid >= rows) return;
    const int kk = (int)(gid / ((int64_t)d.s * d.s));
    const int r = (int)(gid - (int64_t)kk * d.s * d.s);
    const int d1 = r / d.s, d2 = r - d1 * d.s;
    int c[3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
        c[a] = (int)__umul64hi(sm64_draw(d.key, 1u, 3ull * kk + a), (uint64_t)d.n);
    for (int d3 = 0; d3 < d.s; ++d3) mask[d.cell_off + l3(d, c[0] + d1, c[1] + d2, c[2] + d3)] = 1;
}

// ----------------------------------------------------------- stiffness --
// y = A x for one pair.  An entry E[a][b] of the element matrix depends only
// on the number of axes along which the corners a and b differ (K1 and M1
// are symmetric with equal diagonals): e_0 = 3 m0^2 / h, e_1 = (2 m0 m1 -
// m0^2) / h, e_2 = (m1^2 - 2 m0 m1) / h, e_3 = -3 m1^2 / h with M1 = [m0 m1;
// m1 m0].  Consistent (m0 = h/3, m1 = h/6): e_0 = h/3, e_1 = 0, e_2 = e_3 =
// -h/12; lumped (m0 = h/2, m1 = 0): e_0 = 3h/4, e_1 = -h/4, e_2 = e_3 = 0.
// So the assembled row of node i couples neighbour i+o (o in {-1,0,1}^3)
// with e_{|o|} times the sum of a_c over the cells holding both nodes: all 8
// for o = 0, 4 for a face neighbour, 2 for an edge neighbour (a pair sum
// along the axis where o is 0), 1 for a corner neighbour: about 60
// operations per node and pair instead of 144 for the 8 element rows.
// A thread computes two neighbouring nodes (k0, k0 + 1) of one row in SZ
// consecutive planes; a block takes TJ = 512 / n whole rows of those planes.
// It first copies the planes i0-1 .. i0+SZ, rows j0-1 .. j0+TJ of x and the
// cell values of planes i0-1 .. i0+SZ-1, rows j0-1 .. j0+TJ-1 (whole periodic
// rows) into shared memory, every load issued before the first store, then
// each node sums the contributions of its three x-planes: from below (cells
// of plane i-1), in its own plane (both cell planes and the diagonal term)
// and from above (cells of plane i).  Per node pair and row one 16-byte and
// two 8-byte shared loads.
//   MODE_APPLY: y = A x, partials of x.y per component (the p.q of CG);
//   MODE_RESID: y = f - A x (the true residual), partials of |y|^2.
// Blocks of units whose flag (`done`, or `outer_done` for MODE_RESID) is
// set return at once.
enum { MODE_APPLY = 0, MODE_RESID = 1 };
struct MixScal;
__device__ __forceinline__ bool unit_skip(const MixScal* sc, int u, bool outer);

// Shared memory of a stiffness block for grids of n = 2^lg.
template <typename V>
__host__ __device__ constexpr size_t stiff_smem(int lg) {
    return (size_t)(SZ + 2) * (((2 * T3) >> lg) + 2) * ((size_t)1 << lg) * sizeof(V) +
           (size_t)(SZ + 1) * (((2 * T3) >> lg) + 1) * ((size_t)1 << lg) * (sizeof(V) / 2);
}

// Two consecutive elements (16-byte aligned for float2 pairs).
template <typename V> struct Two { V a, b; };
__device__ __forceinline__ Two<float2> ld_two(const float2* p) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ Two<double2> ld_two(const double2* p) { return {p[0], p[1]}; }
__device__ __forceinline__ void st_two(float2* p, const Two<float2>& t) {
    *reinterpret_cast<float4*>(p) = make_float4(t.a.x, t.a.y, t.b.x, t.b.y);
}
__device__ __forceinline__ void st_two(double2* p, const Two<double2>& t) { p[0] = t.a; p[1] = t.b; }
template <typename T> __device__ __forceinline__ Two<T> ld_two_s(const T* p) { return {p[0], p[1]}; }
template <> __device__ __forceinline__ Two<float> ld_two_s<float>(const float* p) {
    const float2 v = *reinterpret_cast<const float2*>(p);
    return {v.x, v.y};
}

// FP32: three blocks per SM (80 registers, no spills) with the register
// window below.
template <int SCHEME, int MODE, typename V>
__global__ void __launch_bounds__(T3, sizeof(V) == 8 ? (SCHEME == RVE_Q1_LUMPED ? 4 : 3) : 2)
    k3_stiffness(Grp g, Cells3T<typename ScalarOf<V>::T> cs, const V* __restrict__ x,
                 V* __restrict__ y, const V* __restrict__ f, double* part, const MixScal* sc) {
    typedef typename ScalarOf<V>::T T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[16];
    int lb;
    const int u = unit_of(g, lb);
    const U3 d = g.desc[u];   // issued before the flag test
    if (sc && unit_skip(sc, u, MODE == MODE_RESID)) return;
    const int n = d.n, m = n - 1, lg = d.log2n;
    const int TJ = (2 * T3) >> lg;                    // rows of the block
    const int first = lb * (2 * T3);                  // (plane group, j0, 0)
    const int i0 = (first >> (2 * lg)) * SZ;
    const int j0 = (first >> lg) & m;
    const int jl = threadIdx.x >> (lg - 1), k0 = 2 * (threadIdx.x & ((n >> 1) - 1));
    const int RW = TJ + 2, CR = TJ + 1;               // rows of the x and cell tiles
    V* xt = reinterpret_cast<V*>(smem_raw);                          // [SZ+2][RW][n]
    T* ct = reinterpret_cast<T*>(xt + (SZ + 2) * RW * n);            // [SZ+1][CR][n]
    const V* __restrict__ xu = x + d.off;
    const T am = two_values<T>(d, false), ai = two_values<T>(d, true);
    const uint8_t* __restrict__ mk8 = cs.mask + d.cell_off;
    const T* __restrict__ cf = cs.coef ? cs.coef + d.cell_off : nullptr;
    // copy: thread (jl, k0) takes elements k0, k0+1 of tile rows jl, jl + TJ
    // (those below RW, resp. CR) of each plane; x by asynchronous 16-byte
    // copies (no registers held), the cell values through registers (they
    // are converted), every load issued before the first store
    constexpr int CHUNKS = (int)(2 * sizeof(V) / 16);   // 16-byte pieces of two elements
#pragma unroll
    for (int pl = 0; pl < SZ + 2; ++pl) {
        const int gp = ((i0 - 1 + pl) & m) << (2 * lg);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int rr = jl + q * TJ;
            if (rr < RW) {
                const char* gsrc = reinterpret_cast<const char*>(xu + gp + (((j0 - 1 + rr) & m) << lg) + k0);
                const unsigned sdst = (unsigned)__cvta_generic_to_shared(xt + (pl * RW + rr) * n + k0);
#pragma unroll
                for (int c = 0; c < CHUNKS; ++c)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sdst + 16 * c),
                                 "l"(gsrc + 16 * c)
                                 : "memory");
            }
        }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    Two<T> cr[SZ + 1][2];
#pragma unroll
    for (int pl = 0; pl < SZ + 1; ++pl) {
        const int gp = ((i0 - 1 + pl) & m) << (2 * lg);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int rr = jl + q * TJ;
            if (rr < CR) {
                const int idx = gp + (((j0 - 1 + rr) & m) << lg) + k0;
                if (cf) {
                    cr[pl][q] = ld_two_s(cf + idx);
                } else {
                    const uchar2 mb = *reinterpret_cast<const uchar2*>(mk8 + idx);
                    cr[pl][q] = {mb.x ? ai : am, mb.y ? ai : am};
                }
            }
        }
    }
#pragma unroll
    for (int pl = 0; pl < SZ + 1; ++pl)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int rr = jl + q * TJ;
            if (rr < CR) {
                T* c = ct + (pl * CR + rr) * n + k0;
                c[0] = cr[pl][q].a;
                c[1] = cr[pl][q].b;
            }
        }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    const int kl = (k0 - 1) & m, kr = (k0 + 2) & m;
    const T h = (T)d.h;
    // the cell bit that a neighbour offset fixes on its axis: +1 -> 0, -1 -> 1
    auto cb = [](int o) { return o > 0 ? 0 : 1; };
    const T e0 = SCHEME == RVE_Q1_CONSISTENT ? h * (T)(1.0 / 3.0) : h * (T)0.75;
    const T eo = SCHEME == RVE_Q1_CONSISTENT ? -h * (T)(1.0 / 12.0) : -h * (T)0.25;
    // C[q]: the cell at (j - c2, k - c3) of a cell plane, q = 2 c2 + c3;
    // X[a][b]: x at (j + a - 1, k + b - 1) of an x-plane
    auto side = [&](const V (&X)[3][3], const T (&C)[4]) -> V {   // off-plane couplings
        T sx = 0, sy = 0;
        if (SCHEME == RVE_Q1_CONSISTENT) {
#pragma unroll
            for (int s2 = -1; s2 <= 1; s2 += 2) {
                const T wy = C[cb(s2)] + C[2 + cb(s2)];           // edge (., 0, s2)
                sx = fma(wy, X[1][1 + s2].x, sx);
                sy = fma(wy, X[1][1 + s2].y, sy);
                const T wz = C[2 * cb(s2)] + C[2 * cb(s2) + 1];   // edge (., s2, 0)
                sx = fma(wz, X[1 + s2][1].x, sx);
                sy = fma(wz, X[1 + s2][1].y, sy);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {                          // corners (., o2, o3)
                const int o2 = (c & 2) ? 1 : -1, o3 = (c & 1) ? 1 : -1;
                const T w = C[2 * cb(o2) + cb(o3)];
                sx = fma(w, X[1 + o2][1 + o3].x, sx);
                sy = fma(w, X[1 + o2][1 + o3].y, sy);
            }
        } else {                                                    // face (., 0, 0)
            const T w = (C[0] + C[1]) + (C[2] + C[3]);
            sx = w * X[1][1].x;
            sy = w * X[1][1].y;
        }
        return mk<V>(eo * sx, eo * sy);
    };
    auto inplane = [&](const V (&X)[3][3], const T (&Cm)[4], const T (&C0)[4]) -> V {
        T px[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) px[q] = Cm[q] + C0[q];
        const T A0 = (px[0] + px[1]) + (px[2] + px[3]);
        T sx = 0, sy = 0;
        if (SCHEME == RVE_Q1_CONSISTENT) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {                          // edges (0, s1, s2)
                const int s1 = (c & 2) ? 1 : -1, s2 = (c & 1) ? 1 : -1;
                const T w = px[2 * cb(s1) + cb(s2)];
                sx = fma(w, X[1 + s1][1 + s2].x, sx);
                sy = fma(w, X[1 + s1][1 + s2].y, sy);
            }
        } else {
#pragma unroll
            for (int sg = -1; sg <= 1; sg += 2) {
                const int v0 = cb(sg);
                const T wj = px[2 * v0] + px[2 * v0 + 1];           // face (0, sg, 0)
                sx = fma(wj, X[1 + sg][1].x, sx);
                sy = fma(wj, X[1 + sg][1].y, sy);
                const T wk = px[v0] + px[2 + v0];                   // face (0, 0, sg)
                sx = fma(wk, X[1][1 + sg].x, sx);
                sy = fma(wk, X[1][1 + sg].y, sy);
            }
        }
        const T dA = e0 * A0;
        return mk<V>(fma(eo, sx, dA * X[1][1].x), fma(eo, sy, dA * X[1][1].y));
    };
    // cells of tile plane pl for the two nodes
    auto cells = [&](int pl, T (&c0)[4], T (&c1)[4]) {
#pragma unroll
        for (int c2 = 0; c2 < 2; ++c2) {
            const T* r = ct + (pl * CR + jl + 1 - c2) * n;
            const Two<T> M = ld_two_s(r + k0);
            const T Lv = r[kl];
            c0[2 * c2] = M.a;       // node k0: c3 = 0 -> k0, c3 = 1 -> k0 - 1
            c0[2 * c2 + 1] = Lv;
            c1[2 * c2] = M.b;       // node k0 + 1: c3 = 0 -> k0 + 1, c3 = 1 -> k0
            c1[2 * c2 + 1] = M.a;
        }
    };
    T dx = 0, dy = 0;
    // adds the couplings through x-plane t + o1 (X0, X1: [row][k] windows of
    // the two nodes) to acc0, acc1; cell planes t - 1 (Cm*) and t (C0*)
    auto couple = [&](int o1, const V (&X0)[3][3], const V (&X1)[3][3], const T (&Cm0)[4],
                      const T (&Cm1)[4], const T (&C00)[4], const T (&C01)[4], V& acc0, V& acc1) {
        V v0, v1;
        if (o1 < 0) { v0 = side(X0, Cm0); v1 = side(X1, Cm1); }
        else if (o1 == 0) { v0 = inplane(X0, Cm0, C00); v1 = inplane(X1, Cm1, C01); }
        else { v0 = side(X0, C00); v1 = side(X1, C01); }
        acc0.x += v0.x; acc0.y += v0.y;
        acc1.x += v1.x; acc1.y += v1.y;
    };
    // output plane t of the two nodes (xa, xb: their own x values)
    auto emit = [&](int t, V acc0, V acc1, const V& xa, const V& xb) {
        const int64_t node = d.off + ((int64_t)(i0 + t) << (2 * lg)) + ((j0 + jl) << lg) + k0;
        if (MODE == MODE_RESID) {
            const Two<V> ff = ld_two(f + node);
            acc0.x = ff.a.x - acc0.x; acc0.y = ff.a.y - acc0.y;
            acc1.x = ff.b.x - acc1.x; acc1.y = ff.b.y - acc1.y;
            dx = fma(acc0.x, acc0.x, fma(acc1.x, acc1.x, dx));
            dy = fma(acc0.y, acc0.y, fma(acc1.y, acc1.y, dy));
        } else {
            dx = fma(xa.x, acc0.x, fma(xb.x, acc1.x, dx));
            dy = fma(xa.y, acc0.y, fma(xb.y, acc1.y, dy));
        }
        st_two(y + node, Two<V>{acc0, acc1});
    };
    if constexpr (sizeof(T) == 4) {
        // FP32: a window of three x-planes (rows jl .. jl + 2, k0 - 1 ..
        // k0 + 2) and two cell planes rolls down the block's planes in
        // registers, so each tile plane is read from shared memory once
        // instead of three times and each cell plane once instead of twice.
        // The arithmetic and its order are those of the FP64 branch.
        V W[3][3][4];
        auto xplane = [&](int pl, V (&P)[3][4]) {
#pragma unroll
            for (int a2 = 0; a2 < 3; ++a2) {
                const V* r = xt + (pl * RW + jl + a2) * n;
                const Two<V> M = ld_two(r + k0);
                P[a2][0] = r[kl];
                P[a2][1] = M.a;
                P[a2][2] = M.b;
                P[a2][3] = r[kr];
            }
        };
        auto step = [&](int t, const T (&Cm0)[4], const T (&Cm1)[4], const T (&C00)[4],
                        const T (&C01)[4]) {
            V acc0 = mk<V>((T)0, (T)0), acc1 = acc0;
#pragma unroll
            for (int o1 = -1; o1 <= 1; ++o1) {
                const V (&P)[3][4] = W[(t + 1 + o1) % 3];
                V X0[3][3], X1[3][3];
#pragma unroll
                for (int a2 = 0; a2 < 3; ++a2)
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        X0[a2][q] = P[a2][q];
                        X1[a2][q] = P[a2][q + 1];
                    }
                couple(o1, X0, X1, Cm0, Cm1, C00, C01, acc0, acc1);
            }
            const V (&P0)[3][4] = W[(t + 1) % 3];
            emit(t, acc0, acc1, P0[1][1], P0[1][2]);
        };
        T Ca0[4], Ca1[4], Cb0[4], Cb1[4];
        xplane(0, W[0]);
        xplane(1, W[1]);
        cells(0, Ca0, Ca1);
#pragma unroll
        for (int t = 0; t < SZ; ++t) {
            xplane(t + 2, W[(t + 2) % 3]);
            if (t % 2 == 0) {
                cells(t + 1, Cb0, Cb1);
                step(t, Ca0, Ca1, Cb0, Cb1);
            } else {
                cells(t + 1, Ca0, Ca1);
                step(t, Cb0, Cb1, Ca0, Ca1);
            }
        }
    } else {
        // FP64: a register window would not fit; each plane step reads its
        // three x-planes and two cell planes from shared memory
#pragma unroll 1
        for (int t = 0; t < SZ; ++t) {
            T Cm0[4], Cm1[4], C00[4], C01[4];
            cells(t, Cm0, Cm1);
            cells(t + 1, C00, C01);
            V acc0 = mk<V>((T)0, (T)0), acc1 = acc0;
#pragma unroll
            for (int o1 = -1; o1 <= 1; ++o1) {
                V X0[3][3], X1[3][3];
#pragma unroll
                for (int a2 = 0; a2 < 3; ++a2) {
                    const V* r = xt + ((t + 1 + o1) * RW + jl + a2) * n;
                    const Two<V> M = ld_two(r + k0);
                    const V Lv = r[kl], Rv = r[kr];
                    X0[a2][0] = Lv;  X0[a2][1] = M.a; X0[a2][2] = M.b;
                    X1[a2][0] = M.a; X1[a2][1] = M.b; X1[a2][2] = Rv;
                }
                couple(o1, X0, X1, Cm0, Cm1, C00, C01, acc0, acc1);
            }
            const Two<V> xc = ld_two(xt + ((t + 1) * RW + jl + 1) * n + k0);
            emit(t, acc0, acc1, xc.a, xc.b);
        }
    }
    if (part) {   // block-uniform
        double tx = 0.0, ty = 0.0;
        block_pair_sum(dx, dy, red, tx, ty);
        if (threadIdx.x == 0) {
            part[d.part_off + 2 * lb] = tx;
            part[d.part_off + 2 * lb + 1] = ty;
        }
    }
}

// ------------------------------------------- double-word true residual --
// The mixed path's true residual r64 = f - A u without FP64 arithmetic per
// node (GB300's FP64 pipe is ~1/64 of FP32): u is split once into double
// words (hi, lo floats from its IEEE fields, k3_split_dw), and the row of
// node i is scaled by K = 12/h (consistent) or 4/h (lumped), which makes
// every Hamming-distance weight an integer multiple of a sum of cell values:
//   consistent  K e = (4, 0, -1, -1)    K r = K f - 4 S8 u_i + sum_edges S2 u + sum_corners S1 u
//   lumped      K e = (3, -1, 0, 0)     K r = K f - 3 S8 u_i + sum_faces S4 u
// (S_m the sum of the m cells the two nodes share).  The sum is a
// compensated dot product of double words (DotDW: the products' rounding
// errors gather in a compensation term), so its absolute error is
// O(eps_32^2) times the size of its terms -- far below the outer tolerance
// -- like the 2D refinement pass.  One node per thread; the neighbours'
// double words come through L1.  Partials: |r|^2 per component (FP32 per
// thread, 256 nodes per block).
__global__ void __launch_bounds__(T3) k3_split_dw(Grp g, const double2* __restrict__ u,
                                                  float4* __restrict__ w, const MixScal* sc) {
    int lb;
    const int un = unit_of(g, lb);
    const U3 d = g.desc[un];
    if (unit_skip(sc, un, true)) return;
    const int64_t node = d.off + (int64_t)lb * T3 + threadIdx.x;
    const double2 v = u[node];
    const dword x = dw_split(v.x), y = dw_split(v.y);
    w[node] = make_float4(x.hi, y.hi, x.lo, y.lo);
}

// EXACT: both cell values are integers of magnitude <= 2^20 (the paper's
// two-valued coefficients), so every cell sum below (at most 8 cells, below
// 2^24) and its power-of-two scalings are exact in one float; the weights
// are then floats instead of double words, with the same values and so the
// same result.
template <int SCHEME, bool EXACT>
__device__ __forceinline__ void resid_dw_body(const U3& d, int lb, Cells3T<double> cs,
                                              const float4* __restrict__ w,
                                              const double2* __restrict__ f,
                                              double2* __restrict__ r, double* part,
                                              double* red) {
    typedef std::conditional_t<EXACT, float, dword> CW;
    auto wadd = [](CW x, CW y) -> CW {
        if constexpr (EXACT) return __fadd_rn(x, y); else return dw_add(x, y);
    };
    auto wneg = [](CW x) -> CW {
        if constexpr (EXACT) return -x; else return dw_neg(x);
    };
    auto wscale2 = [](CW x, float p2) -> CW {
        if constexpr (EXACT) return x * p2; else return dw_scale2(x, p2);
    };
    const int lg = d.log2n;
    const int loc = lb * T3 + threadIdx.x;
    const int i = loc >> (2 * lg), j = (loc >> lg) & (d.n - 1), k = loc & (d.n - 1);
    const float4* __restrict__ wu = w + d.off;
    const dword aI = dw_split(d.ai), aM = dw_split(d.am);
    // the 8 cells around the node: C[4 c1 + 2 c2 + c3] = cell (i - c1, j - c2, k - c3)
    CW C[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int idx = l3(d, i - (q >> 2), j - ((q >> 1) & 1), k - (q & 1));
        if constexpr (EXACT) {   // mask only
            C[q] = __ldg(cs.mask + d.cell_off + idx) ? aI.hi : aM.hi;
        } else {
            if (cs.coef) C[q] = dw_split(__ldg(cs.coef + d.cell_off + idx));
            else C[q] = __ldg(cs.mask + d.cell_off + idx) ? aI : aM;
        }
    }
    // the cell bit an offset fixes on its axis: +1 -> 0, -1 -> 1
    auto cb = [](int o) { return o > 0 ? 0 : 1; };
    // K = 12/h or 4/h: an integer (h = 1/m0)
    const float K = (SCHEME == 0 ? 12.f : 4.f) * rintf((float)(1.0 / d.h));
    const double2 ff = f[d.off + loc];
    DotDW rx(dw_mulf(dw_split(ff.x), K)), ry(dw_mulf(dw_split(ff.y), K));
    auto term = [&](CW wgt, int o1, int o2, int o3) {   // r -= wgt * u(i + o)
        const float4 v = wu[l3(d, i + o1, j + o2, k + o3)];
        const CW nw = wneg(wgt);
        rx.add(nw, v.x, v.z);
        ry.add(nw, v.y, v.w);
    };
    const CW S8 = wadd(wadd(wadd(C[0], C[1]), wadd(C[2], C[3])),
                       wadd(wadd(C[4], C[5]), wadd(C[6], C[7])));
    term(wscale2(S8, SCHEME == 0 ? 4.f : 2.f), 0, 0, 0);
    if (SCHEME != 0) term(S8, 0, 0, 0);   // 3 S8 = 2 S8 + S8 (exact scalings only)
#pragma unroll
    for (int o1 = -1; o1 <= 1; ++o1)
#pragma unroll
        for (int o2 = -1; o2 <= 1; ++o2)
#pragma unroll
            for (int o3 = -1; o3 <= 1; ++o3) {
                const int zeros = (o1 == 0) + (o2 == 0) + (o3 == 0);
                if (zeros == 3) continue;
                if (SCHEME == 0 && zeros == 2) continue;   // faces: K e_1 = 0
                if (SCHEME != 0 && zeros != 2) continue;   // lumped: faces only
                // sum of the cells shared with the neighbour: the bits of
                // the non-zero offsets are fixed, the others run over 0, 1
                CW S{};
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int c1 = q >> 2, c2 = (q >> 1) & 1, c3 = q & 1;
                    if (o1 != 0 && c1 != cb(o1)) continue;
                    if (o2 != 0 && c2 != cb(o2)) continue;
                    if (o3 != 0 && c3 != cb(o3)) continue;
                    S = wadd(S, C[q]);
                }
                term(wneg(S), o1, o2, o3);   // K e = -1: r += S u
            }
    const double invK = 1.0 / (double)K;
    const double rxd = ((double)rx.s + (double)rx.comp) * invK;
    const double ryd = ((double)ry.s + (double)ry.comp) * invK;
    r[d.off + loc] = make_double2(rxd, ryd);
    if (part) {
        const float fx = (float)rxd, fy = (float)ryd;
        double tx = 0.0, ty = 0.0;
        block_pair_sum(fx * fx, fy * fy, red, tx, ty);
        if (threadIdx.x == 0) {
            part[d.part_off + 2 * lb] = tx;
            part[d.part_off + 2 * lb + 1] = ty;
        }
    }
}

template <int SCHEME>
__global__ void __launch_bounds__(T3) k3_resid_dw(Grp g, Cells3T<double> cs,
                                                  const float4* __restrict__ w,
                                                  const double2* __restrict__ f,
                                                  double2* __restrict__ r, double* part,
                                                  const MixScal* sc) {
    __shared__ double red[16];
    int lb;
    const int un = unit_of(g, lb);
    const U3 d = g.desc[un];
    if (unit_skip(sc, un, true)) return;
    auto small_int = [](double a) { return a == floor(a) && fabs(a) <= 1048576.0; };
    if (!cs.coef && small_int(d.ai) && small_int(d.am))
        resid_dw_body<SCHEME, true>(d, lb, cs, w, f, r, part, red);
    else
        resid_dw_body<SCHEME, false>(d, lb, cs, w, f, r, part, red);
}

// -------------------------------------------------------------- loads --
// Corrector loads f_i = -sum_c a_c P_c^T E xi_i (xi_i = h x corner bit i).
// Every row of M1 sums to h/2 (both schemes) and every row of K1 to 0, so
// of the three Kronecker terms only the one with K1 along axis i survives,
// and the row of E xi_i at local corner l is (h^2/4) (+1 if l_i = 1, -1
// otherwise).  Summed over the 8 cells around the node (the node is corner
// c of the cell at offset -c):
//     f_i = (h^2/4) (sum_{c_i = 0} a_c - sum_{c_i = 1} a_c),
// which is exactly zero where the 8 cells agree.  Unit pair 0 gets (f_1,
// f_2), pair 1 gets (f_3, 0).  Also the partials of |f|^2.
__global__ void __launch_bounds__(T3) k3_rhs(Grp g, Cells3T<double> cs, double2* __restrict__ f,
                                             double* part) {
    __shared__ double red[32];
    int lb;
    const int u = unit_of(g, lb);
    const U3& d = g.desc[u];
    const int local = lb * T3 + threadIdx.x;
    const int n = d.n;
    const int i = local >> (2 * d.log2n), j = (local >> d.log2n) & (n - 1), k = local & (n - 1);
    double a[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const int idx = l3(d, i - (c >> 2), j - ((c >> 1) & 1), k - (c & 1));
        a[c] = cs.coef ? cs.coef[d.cell_off + idx] : two_values<double>(d, cs.mask[d.cell_off + idx] != 0);
    }
    const double q = 0.25 * d.h * d.h;
    double2 out;
    if (d.pair == 0) {   // cells summed along the third axis, then differences along the first two
        const double t00 = a[0] + a[1], t01 = a[2] + a[3], t10 = a[4] + a[5], t11 = a[6] + a[7];
        out = make_double2(q * ((t00 + t01) - (t10 + t11)), q * ((t00 + t10) - (t01 + t11)));
    } else {
        out = make_double2(q * (((a[0] + a[2]) + (a[4] + a[6])) - ((a[1] + a[3]) + (a[5] + a[7]))), 0.0);
    }
    f[d.off + local] = out;
    if (part) {
        DotAcc<double> dx, dy;
        dx.add(out.x, out.x);
        dy.add(out.y, out.y);
        double tx = 0.0, ty = 0.0;
        block_sum2(dx, dy, red, tx, ty);
        if (threadIdx.x == 0) {
            part[d.part_off + 2 * lb] = tx;
            part[d.part_off + 2 * lb + 1] = ty;
        }
    }
}

// ------------------------------------------------------ preconditioner --
// Hartley transform of lines of n nodes (pair-packed complex FFT, register
// Stockham, see rve_device.cuh): dst = scale H src (src may equal dst).
// AXIS 2: x lines (contiguous), threads of a line side by side, one padded
// buffer per line; AXIS 1: y lines (stride n), the G lines of a block side
// by side so that each load instruction reads consecutive nodes, and their
// buffers interleaved element by element so that the lanes of a warp (G
// consecutive lines at the same element) touch consecutive words.
//
// STEP: the last x pass of a CG step, which forms the new direction from the
// preconditioned residual without storing it: with p the old direction, e +=
// alpha p and p = scale H src + beta p (e and p are the step's, src is left).
// r.z, and so beta, comes from the z solve one pass earlier.  Before, the pass
// stored z and read r for r.z, a launch formed p = z + beta p, and e += alpha p
// read p beside the residual's update: 177 bytes per node and step in FP32,
// 145 now; 15 realizations of 64^3 37.4 -> 33.2 ms.
// Double pairs are transformed in fixed point (rve_fixed.cuh, as the 2D rows
// are), the block's lines all of them or, where one cannot be, all in FP64.
template <typename T> __device__ __forceinline__ T alpha_of(const MixScal& s, int k);
template <typename T> __device__ __forceinline__ T beta_of(const MixScal& s, int k);
template <int LOG2N, int BS>
__device__ __noinline__ void hartley_line_fp64(double2* w, double2* buf, int t, const double2* __restrict__ tw) {
    constexpr int n = 1 << LOG2N, TL = n / 8;
    double2 v[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) v[m] = w[m];
    fft_reg<FFT_TO_BOTH, LOG2N, BS>(v, buf, LOG2N, t, tw, true);
#pragma unroll
    for (int m = 0; m < 8; ++m) w[m] = hartley_pair(v[m], buf[pidx((n - (t + m * TL)) & (n - 1)) * BS]);
}
// w[m] = element t + m TL of line q -> of its Hartley transform; `ex` (shared):
// two words per line of the block.
template <int LOG2N, int BS>
__device__ __forceinline__ void hartley_line(double2 (&w)[8], double2* buf, int q, int t, const Tables& tb,
                                             unsigned* ex) {
    constexpr int n = 1 << LOG2N, TL = n / 8, G = 256 / TL;
    if (threadIdx.x < 2 * G) ex[threadIdx.x] = 0u;
    unsigned hi = 0;
#pragma unroll
    for (int m = 0; m < 8; ++m)
        hi = max(hi, max((unsigned)__double2hiint(w[m].x) & 0x7FFFFFFFu, (unsigned)__double2hiint(w[m].y) & 0x7FFFFFFFu));
    if (hi == 0u) {   // zeros, or subnormals (which count as 1)
#pragma unroll
        for (int m = 0; m < 8; ++m)
            hi |= fx_high(0u, (unsigned)__double2loint(w[m].x) | (unsigned)__double2loint(w[m].y));
    }
    __syncthreads();
    atomicMax(ex + q, hi);
    __syncthreads();
    unsigned E = fx_row_exponent(ex[q]);
    if (LOG2N >= 7 && fx_takes(E)) {
        unsigned s = 0;
#pragma unroll
        for (int m = 0; m < 8; ++m)
            s += fx_size((unsigned)__double2hiint(w[m].x), E) + fx_size((unsigned)__double2hiint(w[m].y), E);
        atomicAdd(ex + G + q, s);
    }
    if (__syncthreads_and(fx_takes(E))) {
        FxTw fx = fx_twiddles(tb, n);
        fx.f = fx_schedule(LOG2N, ex[G + q]);
        E -= fx.f.finer;
        longlong2 f[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) f[m] = make_longlong2(fx_from(w[m].x, E), fx_from(w[m].y, E));
        longlong2* fb = reinterpret_cast<longlong2*>(buf);
        fft_reg<FFT_TO_BOTH, LOG2N, BS>(f, fb, LOG2N, t, fx, true);
        const int e = (int)E - FX_BITS + fx_scale(LOG2N, fx.f) - 1;   // the pairs come doubled
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const longlong2 h = hartley_pair2(f[m], fb[pidx((n - (t + m * TL)) & (n - 1)) * BS]);
            w[m] = make_double2(fx_to(h.x, e), fx_to(h.y, e));
        }
    } else {
        double2 v[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) v[m] = w[m];
        hartley_line_fp64<LOG2N, BS>(v, buf, t, twiddles<double2>(tb, n));
#pragma unroll
        for (int m = 0; m < 8; ++m) w[m] = v[m];
    }
}
template <int LOG2N, int AXIS, bool STEP, typename V>
__global__ void __launch_bounds__(256) k3_lines(Grp g, Tables tb, const V* src, V* dst,
                                                typename ScalarOf<V>::T scale, V* __restrict__ e,
                                                const MixScal* sc) {
    typedef typename ScalarOf<V>::T T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned ex[sizeof(V) == 16 ? 2 * 256 * 8 / (1 << LOG2N) : 1];
    int lb;
    const int u = unit_of(g, lb);
    const U3 d = g.desc[u];   // issued before the flag test
    if (sc && unit_skip(sc, u, false)) return;
    constexpr int n = 1 << LOG2N, TL = n / 8, G = 256 / TL;
    constexpr int BS = AXIS == 2 ? 1 : G;
    int q, t;
    if (AXIS == 2) { q = threadIdx.x / TL; t = threadIdx.x - q * TL; }
    else { t = threadIdx.x / G; q = threadIdx.x - t * G; }
    const int line = lb * G + q;   // < n^2
    int64_t base, stride;
    if (AXIS == 2) { base = d.off + (int64_t)line * n; stride = 1; }
    else { base = d.off + (int64_t)(line / n) * n * n + (line % n); stride = n; }
    V* buf = reinterpret_cast<V*>(smem_raw) + (AXIS == 2 ? q * seq_stride(n) : q);
    V w[8];
#pragma unroll
    for (int mm = 0; mm < 8; ++mm) w[mm] = src[base + (t + mm * TL) * stride];
    if constexpr (sizeof(V) == 16) hartley_line<LOG2N, BS>(w, buf, q, t, tb, ex);
    else fft_reg<FFT_TO_BOTH, LOG2N, BS>(w, buf, LOG2N, t, twiddles<V>(tb, n), true);
    T ax = 0, ay = 0, bx = 0, by = 0;
    if (STEP) {
        ax = alpha_of<T>(sc[u], 0);
        ay = alpha_of<T>(sc[u], 1);
        bx = beta_of<T>(sc[u], 0);
        by = beta_of<T>(sc[u], 1);
    }
    // in halves of four: a half's loads before its stores
#pragma unroll
    for (int h = 0; h < 8; h += 4) {
        V po[4], eo[4];
        if (STEP) {
#pragma unroll
            for (int mm = 0; mm < 4; ++mm) {
                const int64_t node = base + (int64_t)(t + (h + mm) * TL) * stride;
                po[mm] = dst[node];
                eo[mm] = e[node];
            }
        }
#pragma unroll
        for (int mm = 0; mm < 4; ++mm) {
            const int kx = t + (h + mm) * TL;
            const int64_t node = base + (int64_t)kx * stride;
            V hv = w[h + mm];   // FP64: transformed by hartley_line
            if constexpr (sizeof(V) == 8) hv = hartley_pair(hv, buf[pidx((n - kx) & (n - 1)) * BS]);
            V o = mk<V>(scale * hv.x, scale * hv.y);
            if (STEP) {
                e[node] = mk<V>(fma(ax, po[mm].x, eo[mm].x), fma(ay, po[mm].y, eo[mm].y));
                o = mk<V>(fma(bx, po[mm].x, o.x), fma(by, po[mm].y, o.y));
            }
            dst[node] = o;
        }
    }
}

// Tridiagonal solves along z after the x and y transforms; writes M^{-1} t
// / n in place and, with `part`, the partials of r.z (the transforms being
// orthogonal up to n, r.z is a sum over the transformed residual).  The n^2 columns (kx, ky) of a unit are numbered kc = ky n +
// kx, so column kc, row r sits at r n^2 + kc; a block takes ZC consecutive
// columns (ZSEG rows per thread, ZC x n / ZSEG = 512 threads).  The filter
// root of (kx, ky) solves rho + 1/rho = 2 + lambda(kx) + lambda(ky) + delta
// / c0, evaluated in the vector's precision; column 0 with delta = 0 is the
// singular one.
constexpr int ZSEG = 16;
template <int LOG2N> __host__ __device__ constexpr int zcols() { return Z_THREADS / ((1 << LOG2N) / ZSEG); }
template <typename T> __device__ __forceinline__ T filter_root_t(T mu) {
    return (T)1 / ((T)1 + (T)0.5 * mu + sqrt(mu * ((T)1 + (T)0.25 * mu)));
}
template <int LOG2N, typename V>
__global__ void __launch_bounds__(Z_THREADS) k3_zsolve(Grp g, Tables tb, double delta,
                                                       V* __restrict__ v, double* part,
                                                       const MixScal* sc) {
    typedef typename ScalarOf<V>::T T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[64];
    __shared__ T csc[1];
    double pz[2] = {0.0, 0.0};   // thread 0: the block's share of t.(M^-1 t / n)
    int lb;
    const int u = unit_of(g, lb);
    const U3 d = g.desc[u];   // issued before the flag test
    if (sc && unit_skip(sc, u, false)) return;
    constexpr int n = 1 << LOG2N, NN = n * n, ZC = zcols<LOG2N>();
    RDesc cd;          // the two fields the column solve reads
    cd.tC = ZC;
    cd.c0 = d.c0;
    const int c0 = lb * ZC;
    const T* lapT = lap_table<T>(tb, n);
    const T dc = (T)(delta / d.c0);
    V* vu = v + d.off;
    col_solve_core<V, LOG2N, true, ZSEG>(
        [&](int r, int kc) { return vu[r * NN + kc]; },
        [&](int r, int kc, V val) { vu[r * NN + kc] = val; },
        [&](int kc) -> T {
            const int ky = kc >> LOG2N, kx = kc & (n - 1);
            return (ky == 0 && delta == 0.0) ? rho_table<T>(tb, n)[kx]
                                             : filter_root_t<T>(lapT[kx] + lapT[ky] + dc);
        },
        cd, c0, reinterpret_cast<V*>(smem_raw), tb, delta, red, part ? pz : nullptr, csc);
    if (part && threadIdx.x == 0) {   // r.z = t.(M^-1 t / n) / n, t = Hy Hx r
        part[d.part_off + 2 * lb] = pz[0] / (double)n;
        part[d.part_off + 2 * lb + 1] = pz[1] / (double)n;
    }
}

// ------------------------------------------------------------- A_hom --
// Per tile of 4 T3 cells, partial sums of sum a_c, the energy terms
// a_c v_i^T E v_j (ij = 11 12 13 22 23 33) and the flux terms a_c int_c
// d_j (x_i + phi_i) (ij = 11 12 13 21 22 23 31 32 33), v_i = xi_i + P_c u_i.
// The element matrix is diagonal in the sum / difference basis of each axis
// (K1 has 0 and 2/h, M1 has h/2 and h/6, lumped h/2), so with w the 8 signed
// sums of a cell's corner values
//     v^T E v' = (1/8) sum_b lambda_|b| w_b w'_b,   lambda = 0, h/2, h/3, h/6
// (lumped 0, h/2, h, 3h/2), and int_c d_j v = (h^2/4) w_{e_j}.  A thread walks
// up four planes, so that a plane's sums serve two cells: 128 FP64 operations
// per cell instead of 700 with the 8 x 8 products; 15 x 64^3 cells 3.2 -> 1.0 ms.
// Launched over realizations (the pair-0 unit descriptors); u is the ABI
// layout [nodes][3].
constexpr int A3_NP = 16, A3_PLANES = 4;
template <int SCHEME>
__global__ void __launch_bounds__(T3) k3_a_hom_part(Grp g, Cells3T<double> cs,
                                                    const double* __restrict__ u3,
                                                    double* __restrict__ part) {
    __shared__ double red[T3 / 32][A3_NP];
    int lb;
    const int un = unit_of(g, lb);
    const U3& d = g.desc[un];
    const int lg = d.log2n, n = d.n;
    const int first = lb * T3;   // (plane group, j, k)
    const int i0 = (first >> (2 * lg)) * A3_PLANES;
    const int jk = (first & ((1 << (2 * lg)) - 1)) + threadIdx.x;
    const int j = jk >> lg, k = jk & (n - 1);
    const double h = d.h;
    const double* __restrict__ uu = u3 + 3 * d.cell_off;
    // sum, k-, j- and jk-difference of a plane's four corners, per corrector
    auto plane = [&](int i, double (&P)[3][4]) {
        const int64_t a = 3 * (int64_t)l3(d, i, j, k), b = 3 * (int64_t)l3(d, i, j, k + 1);
        const int64_t c = 3 * (int64_t)l3(d, i, j + 1, k), e = 3 * (int64_t)l3(d, i, j + 1, k + 1);
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            const double u00 = uu[a + x], u01 = uu[b + x], u10 = uu[c + x], u11 = uu[e + x];
            const double p0 = u00 + u01, p1 = u10 + u11, q0 = u01 - u00, q1 = u11 - u10;
            P[x][0] = p0 + p1;
            P[x][1] = q0 + q1;
            P[x][2] = p1 - p0;
            P[x][3] = q1 - q0;
        }
    };
    const double l1 = h / 16.0, l2 = SCHEME == 0 ? h / 24.0 : h / 8.0, l3_ = SCHEME == 0 ? h / 48.0 : 3.0 * h / 16.0;
    double val[A3_NP];
#pragma unroll
    for (int q = 0; q < A3_NP; ++q) val[q] = 0.0;
    double P[3][4];
    plane(i0, P);
#pragma unroll 1
    for (int i = i0; i < i0 + A3_PLANES; ++i) {
        const int cell = l3(d, i, j, k);
        const double a = cs.coef ? cs.coef[d.cell_off + cell] : two_values<double>(d, cs.mask[d.cell_off + cell] != 0);
        double N[3][4], w[3][7];   // w: k, j, i, jk, ik, ij, ijk
        plane(i + 1, N);
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            w[x][0] = P[x][1] + N[x][1];
            w[x][1] = P[x][2] + N[x][2];
            w[x][2] = N[x][0] - P[x][0];
            w[x][3] = P[x][3] + N[x][3];
            w[x][4] = N[x][1] - P[x][1];
            w[x][5] = N[x][2] - P[x][2];
            w[x][6] = N[x][3] - P[x][3];
            w[x][2 - x] += 4.0 * h;   // xi_x
#pragma unroll
            for (int q = 0; q < 4; ++q) P[x][q] = N[x][q];
        }
        const double a1 = a * l1, a2 = a * l2, a3 = a * l3_;
        val[0] += a;
        int q = 1;
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            double s[7];
#pragma unroll
            for (int b = 0; b < 7; ++b) s[b] = (b < 3 ? a1 : b < 6 ? a2 : a3) * w[x][b];
#pragma unroll
            for (int y = x; y < 3; ++y) {
#pragma unroll
                for (int b = 0; b < 7; ++b) val[q] = fma(s[b], w[y][b], val[q]);
                ++q;
            }
        }
#pragma unroll
        for (int x = 0; x < 3; ++x)
#pragma unroll
            for (int y = 0; y < 3; ++y) {
                val[q] = fma(a, w[x][2 - y], val[q]);
                ++q;
            }
    }
#pragma unroll
    for (int q = 7; q < A3_NP; ++q) val[q] *= 0.25 * h * h;
    // the 16 sums over the warp in 16 additions per lane: at each step half of
    // the lanes keep half of the sums; lane l ends with sum bit-reverse(l / 2)
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int w = 8, o = 16; w >= 1; w >>= 1, o >>= 1) {
        const bool hi = lane & o;
#pragma unroll
        for (int q = 0; q < w; ++q) {
            const double send = hi ? val[q] : val[q + w], keep = hi ? val[q + w] : val[q];
            val[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    val[0] += __shfl_xor_sync(0xffffffffu, val[0], 1);
    if (!(lane & 1)) red[wid][((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 + ((lane >> 1) & 1)] = val[0];
    __syncthreads();
    if (threadIdx.x < A3_NP) {
        double t = 0.0;
        for (int w = 0; w < T3 / 32; ++w) t += red[w][threadIdx.x];
        part[d.part_off + (int64_t)lb * A3_NP + threadIdx.x] = t;
    }
}

// One block per realization, a warp per sum (in tile order), then A.
__global__ void __launch_bounds__(512) k3_a_hom_final(Grp g, const double* __restrict__ part,
                                                      double* __restrict__ A, double* __restrict__ Af) {
    __shared__ double s[A3_NP];
    const int un = g.first + blockIdx.x;
    const U3& d = g.desc[un];
    const int b = d.real;
    const int tiles = (int)(((int64_t)d.n * d.n * d.n) / (A3_PLANES * T3));
    const int p = threadIdx.x >> 5;
    const double t = warp_sum_array(part + d.part_off + p, tiles, A3_NP);
    if ((threadIdx.x & 31) == 0) s[p] = t * d.inv_vol;
    __syncthreads();
    if (threadIdx.x >= 9) return;
    const int x = threadIdx.x / 3, y = threadIdx.x % 3;
    const int lo = min(x, y), hi = max(x, y);
    A[9 * (int64_t)b + threadIdx.x] = s[1 + (lo == 0 ? hi : lo + hi + 1)];   // 11 12 13 22 23 33
    if (Af) Af[9 * (int64_t)b + threadIdx.x] = s[7 + threadIdx.x];
}

// ------------------------------------- layout: ABI triples <-> unit pairs --
// Launched over units: unit pair 0 <-> components (1, 2), pair 1 <-> (3, -).
__global__ void __launch_bounds__(T3) k3_split(Grp g, const double* __restrict__ x3,
                                               double2* __restrict__ v) {
    int lb;
    const int un = unit_of(g, lb);
    const U3& d = g.desc[un];
    const int local = lb * T3 + threadIdx.x;
    const int64_t c = 3 * (d.cell_off + local);
    v[d.off + local] = d.pair == 0 ? make_double2(x3[c], x3[c + 1]) : make_double2(x3[c + 2], 0.0);
}

__global__ void __launch_bounds__(T3) k3_join(Grp g, const double2* __restrict__ v,
                                              double* __restrict__ x3) {
    int lb;
    const int un = unit_of(g, lb);
    const U3& d = g.desc[un];
    const int local = lb * T3 + threadIdx.x;
    const int64_t c = 3 * (d.cell_off + local);
    const double2 w = v[d.off + local];
    if (d.pair == 0) { x3[c] = w.x; x3[c + 1] = w.y; }
    else x3[c + 2] = w.x;
}

// Cell values as FP32 for the mixed path's stencil.
__global__ void k3_coef32(const double* __restrict__ coef, float* __restrict__ c32, int64_t count) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) c32[i] = (float)coef[i];
}

// ---------------------------------------------------------- CG cycles --
// Solver state of one unit (device; written by k3_scalar only).
struct MixScal {
    double fnorm[2];    // |f_c|
    double rn_prev[2];  // |r64_c| of the previous refinement
    double s[2];        // scale of the cycle's system (= |r64_c|)
    double target[2];   // relative residual target of the cycle
    double rho[2], alpha[2], beta[2];
    double relres[2];   // last FP64 true relative residual
    float alpha_f[2], beta_f[2], inv_s_f[2];
    int32_t active[2];  // the cycle still iterates on the component
    int32_t cdone[2];   // met the outer tolerance (or f_c = 0), or failed
    int32_t iters[2];
    int32_t stall[2];   // consecutive refinements without a 10x reduction
    int32_t refinements, status;
    int32_t done;       // no component active in the cycle
    int32_t outer_done; // every component finished
};
__device__ __forceinline__ bool unit_skip(const MixScal* sc, int u, bool outer) {
    return outer ? sc[u].outer_done != 0 : sc[u].done != 0;
}
enum { M_FNORM = 0, M_REFINE, M_RHO0, M_ALPHA, M_CONV, M_BETA };
constexpr int MAX_REFINE = 100;
constexpr int MAX_STALL = 4;

// The scalar steps: one block per unit reduces the unit's partial pairs (n^3
// >> pshift of them: one per block of the kernel that wrote them) in a fixed
// order (four warps per component, per-thread strided sums, then the warp tree)
// and threads 0 and 1 apply `what`, one component each: FP64 square roots and
// divisions cost about a microsecond each.  `tfac`: the cycle target is
// max(tfac tol |f| / |r64|, inner_tol).
struct ScalArgs {
    double tol, inner_tol, tfac;
    int max_iter;
};
__global__ void __launch_bounds__(256) k3_scalar(int first, const U3* __restrict__ desc,
                                                 MixScal* scs,
                                                 const double* __restrict__ part, int what,
                                                 int pshift, ScalArgs a) {
    __shared__ double red[8];
    const int u = first + blockIdx.x;
    MixScal* sc = scs + u;
    const U3& d = desc[u];
    if (what != M_FNORM && what != M_REFINE && sc->done) return;
    if (what == M_REFINE && sc->outer_done) return;
    const int nb = (int)(((int64_t)d.n * d.n * d.n) >> pshift);   // partial pairs written
    const double* pp = part + d.part_off + (threadIdx.x >> 7);
    double t = 0.0;
    for (int j = threadIdx.x & 127; j < nb; j += 128) t += pp[2 * j];
    t = warp_sum(t);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x >= 2) return;
    const int k = threadIdx.x;
    const double v = (red[4 * k] + red[4 * k + 1]) + (red[4 * k + 2] + red[4 * k + 3]);
    auto both = [](bool x) { return __all_sync(3u, x) != 0; };
    int status = RVE_OK;   // of this component, where the step sets one
    bool open;
    switch (what) {
        case M_FNORM: {
            const double fn = sqrt(v);
            const bool none = !(v > 0.0);
            sc->fnorm[k] = fn;
            sc->cdone[k] = none;
            sc->active[k] = 0;
            sc->iters[k] = 0;
            sc->stall[k] = 0;
            sc->relres[k] = 0.0;
            sc->rn_prev[k] = fn;
            const bool all = both(none);
            if (k == 0) {
                sc->refinements = 0;
                sc->status = RVE_OK;
                sc->done = 1;
                sc->outer_done = all;
            }
            break;
        }
        case M_REFINE: {
            const int refs = sc->refinements + 1;
            __syncwarp(3u);
            sc->alpha[k] = sc->beta[k] = 0.0;
            sc->alpha_f[k] = sc->beta_f[k] = 0.f;
            sc->inv_s_f[k] = 0.f;
            bool done = sc->cdone[k] != 0;
            open = false;
            if (!done) {
                const double rn = sqrt(v);
                sc->relres[k] = rn / sc->fnorm[k];
                if (!isfinite(rn)) {
                    status = RVE_ENAN;
                    done = true;
                } else if (rn <= a.tol * sc->fnorm[k]) {
                    done = true;
                } else {
                    const int stall = (rn > 0.1 * sc->rn_prev[k]) ? sc->stall[k] + 1 : 0;
                    sc->stall[k] = stall;
                    if (sc->iters[k] >= a.max_iter || refs > MAX_REFINE || stall >= MAX_STALL) {
                        status = RVE_ENOCONV;
                        done = true;
                    } else {
                        sc->rn_prev[k] = rn;
                        sc->s[k] = rn;
                        sc->inv_s_f[k] = (float)(1.0 / rn);
                        sc->target[k] = fmax(a.tfac * a.tol * sc->fnorm[k] / rn, a.inner_tol);
                        open = true;
                    }
                }
            }
            sc->cdone[k] = done;
            sc->active[k] = open;
            const bool all = both(done), idle = both(!open);
            if (k == 0) {
                sc->refinements = refs;
                sc->outer_done = all;
                sc->done = idle;
            }
            break;
        }
        case M_RHO0:
            sc->rho[k] = v;
            break;
        case M_ALPHA: {
            const bool act = sc->active[k] != 0;
            const double al = act ? sc->rho[k] / v : 0.0;
            sc->alpha[k] = al;
            sc->alpha_f[k] = (float)al;
            if (act) sc->iters[k] += 1;
            break;
        }
        case M_CONV: {   // the cycle's residual starts at norm 1
            open = sc->active[k] != 0;
            if (open) {
                const double rn = sqrt(v);
                if (!isfinite(rn)) {
                    status = RVE_ENAN;
                    open = false;
                    sc->cdone[k] = 1;
                } else if (rn <= sc->target[k] || sc->iters[k] >= a.max_iter) {
                    open = false;
                }
                sc->active[k] = open;
            }
            const bool idle = both(!open);
            if (k == 0) sc->done = idle;
            break;
        }
        case M_BETA: {
            const double be = sc->active[k] ? v / sc->rho[k] : 0.0;
            sc->beta[k] = be;
            sc->beta_f[k] = (float)be;
            sc->rho[k] = v;
            break;
        }
    }
    const int st0 = __shfl_sync(3u, status, 0), st1 = __shfl_sync(3u, status, 1);
    if (k == 0 && (st0 != RVE_OK || st1 != RVE_OK)) sc->status = st1 != RVE_OK ? st1 : st0;
}

// The step scalars in the cycle's precision.
template <> __device__ __forceinline__ double alpha_of<double>(const MixScal& s, int k) { return s.alpha[k]; }
template <> __device__ __forceinline__ float alpha_of<float>(const MixScal& s, int k) { return s.alpha_f[k]; }
template <> __device__ __forceinline__ double beta_of<double>(const MixScal& s, int k) { return s.beta[k]; }
template <> __device__ __forceinline__ float beta_of<float>(const MixScal& s, int k) { return s.beta_f[k]; }

// Start of a cycle: r = r64 / s, e = 0, p = 0 (components not iterating: 0).
template <typename V>
__global__ void __launch_bounds__(T3) k3_start(Grp g, const MixScal* scs,
                                               const double2* __restrict__ r64, V* __restrict__ r,
                                               V* __restrict__ e, V* __restrict__ p) {
    typedef typename ScalarOf<V>::T T;
    int lb;
    const int u = unit_of(g, lb);
    const U3 d = g.desc[u];   // issued before the flag test
    const MixScal& sc = scs[u];
    if (sc.done) return;
    const int64_t node = d.off + lb * T3 + threadIdx.x;
    const double2 rr = r64[node];
    V o;
    if (sizeof(T) == 8) {
        o.x = (T)(sc.active[0] ? rr.x / sc.s[0] : 0.0);
        o.y = (T)(sc.active[1] ? rr.y / sc.s[1] : 0.0);
    } else {
        o.x = (T)rr.x * (T)sc.inv_s_f[0];
        o.y = (T)rr.y * (T)sc.inv_s_f[1];
    }
    r[node] = o;
    e[node] = mk<V>((T)0, (T)0);
    p[node] = mk<V>((T)0, (T)0);
}

// r -= alpha q; partials |r|^2.  Four nodes per thread.  (e += alpha p follows
// in the step's last line pass, which reads p anyway.)
template <typename V>
__global__ void __launch_bounds__(T3) k3_update(Grp g, const MixScal* scs, V* __restrict__ r,
                                                const V* __restrict__ q, double* part) {
    typedef typename ScalarOf<V>::T T;
    __shared__ double red[16];
    int lb;
    const int u = unit_of(g, lb);
    const U3 d = g.desc[u];   // issued before the flag test
    const MixScal& sc = scs[u];
    if (sc.done) return;
    const T ax_ = alpha_of<T>(sc, 0), ay_ = alpha_of<T>(sc, 1);
    T sx = 0, sy = 0;
    V qq[4], rr[4];
#pragma unroll
    for (int mm = 0; mm < 4; ++mm) {
        const int64_t node = d.off + (int64_t)lb * (4 * T3) + mm * T3 + threadIdx.x;
        qq[mm] = q[node];
        rr[mm] = r[node];
    }
#pragma unroll
    for (int mm = 0; mm < 4; ++mm) {
        const int64_t node = d.off + (int64_t)lb * (4 * T3) + mm * T3 + threadIdx.x;
        rr[mm].x = fma(-ax_, qq[mm].x, rr[mm].x);
        rr[mm].y = fma(-ay_, qq[mm].y, rr[mm].y);
        r[node] = rr[mm];
        sx = fma(rr[mm].x, rr[mm].x, sx);
        sy = fma(rr[mm].y, rr[mm].y, sy);
    }
    double tx = 0.0, ty = 0.0;
    block_pair_sum(sx, sy, red, tx, ty);
    if (threadIdx.x == 0) {
        part[d.part_off + 2 * lb] = tx;
        part[d.part_off + 2 * lb + 1] = ty;
    }
}

// End of a cycle: u += s (e + alpha p) (components that iterated; the last
// step's alpha p is still due: a unit that is done skips the line pass, and
// alpha is 0 for a component that ended before).
template <typename V>
__global__ void __launch_bounds__(T3) k3_accum(Grp g, const MixScal* scs, const V* __restrict__ e,
                                               const V* __restrict__ p, double2* __restrict__ uv) {
    typedef typename ScalarOf<V>::T T;
    int lb;
    const int u = unit_of(g, lb);
    const U3 d = g.desc[u];   // issued before the flag test
    const MixScal& sc = scs[u];
    if (sc.outer_done) return;
    const int64_t node = d.off + lb * T3 + threadIdx.x;
    const double sx = sc.cdone[0] ? 0.0 : sc.s[0], sy = sc.cdone[1] ? 0.0 : sc.s[1];
    V ee = e[node];
    const V pp = p[node];
    ee.x = fma(alpha_of<T>(sc, 0), pp.x, ee.x);
    ee.y = fma(alpha_of<T>(sc, 1), pp.y, ee.y);
    double2 w = uv[node];
    w.x = fma(sx, (double)ee.x, w.x);
    w.y = fma(sy, (double)ee.y, w.y);
    uv[node] = w;
}

// Per realization: the report of its two units (u_of[b]: the pair-0 unit).
__global__ void k3_report(const MixScal* scs, const U3* __restrict__ desc,
                          const int32_t* __restrict__ u_of, int batch, rve3_solve_info* info) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= batch) return;
    const int u0 = u_of[b];
    const MixScal& s12 = scs[u0];
    const MixScal& s3 = scs[desc[u0].partner];
    rve3_solve_info r;
    r.iters[0] = s12.iters[0];
    r.iters[1] = s12.iters[1];
    r.iters[2] = s3.iters[0];
    r.status = s12.status != RVE_OK ? s12.status : s3.status;
    r.refinements = s12.refinements + s3.refinements;
    r.reserved = 0;
    r.relres[0] = s12.relres[0];
    r.relres[1] = s12.relres[1];
    r.relres[2] = s3.relres[0];
    info[b] = r;
}

// ------------------------------------------------------------ profile --
// Event timing of every 3D launch by kind (diagnostics, enabled together
// with the fused solver's profiler by rve_profile_enable; process-wide, not
// thread-safe): 0 stiffness of the CG steps, 1 line transform (x or y),
// 2 z solve, 3 vector steps of CG (dots, updates), 4 scalar steps (one block
// per unit), 5 FP64 true residual (the stiffness with the residual fused).
enum { P3_STIFF = 0, P3_LINES, P3_ZSOLVE, P3_VECTOR, P3_SCALAR, P3_RESID, P3_K };
struct Prof3 {
    double ms[P3_K] = {};
    long long launches[P3_K] = {};
    std::vector<cudaEvent_t> pool;
    struct Rec { int kind; cudaEvent_t a, b; };
    std::vector<Rec> pending;
    cudaEvent_t get() {
        if (!pool.empty()) {
            cudaEvent_t e = pool.back();
            pool.pop_back();
            return e;
        }
        cudaEvent_t e = nullptr;
        return cudaEventCreate(&e) == cudaSuccess ? e : nullptr;
    }
    void harvest() {   // stream already synchronised
        for (const Rec& r : pending) {
            float t = 0.f;
            if (cudaEventElapsedTime(&t, r.a, r.b) == cudaSuccess) {
                ms[r.kind] += t;
                launches[r.kind] += 1;
            }
            pool.push_back(r.a);
            pool.push_back(r.b);
        }
        pending.clear();
    }
};
static Prof3 g_prof3;

// Brackets the launches issued during its lifetime with two events.
struct Span3 {
    int kind;
    cudaStream_t s;
    cudaEvent_t a = nullptr;
    Span3(cudaStream_t s_, int k) : kind(k), s(s_) {
        if (profile_on() && (a = g_prof3.get()) != nullptr) cudaEventRecord(a, s);
    }
    ~Span3() {
        if (!a) return;
        cudaEvent_t b = g_prof3.get();
        if (!b) { g_prof3.pool.push_back(a); return; }
        cudaEventRecord(b, s);
        g_prof3.pending.push_back({kind, a, b});
    }
};

static void prof3_sync(cudaStream_t s) {
    if (profile_on() && !g_prof3.pending.empty() && cudaStreamSynchronize(s) == cudaSuccess)
        g_prof3.harvest();
}

// ---------------------------------------------------------------- host --
constexpr int N3_MIN = 32, N3_MAX = 256;
constexpr int NVEC = 8;   // unit vectors: f, u, r64, and the cycle's r, z, p, e, q

// The units of one grid size: ids first .. first + count - 1, the pair-0
// units (one per realization) first.
struct Group3 {
    int log2n = 0;
    int first = 0;
    int count = 0;
};

struct Plan3 {
    int batch = 0;
    std::vector<U3> desc;      // 2 * batch units, grouped by size
    std::vector<int32_t> u_of; // pair-0 unit of each realization
    std::vector<Group3> groups;
    int64_t nodes = 0;         // realization nodes (sum n^3)
    int64_t unit_nodes = 0;    // 2 * nodes
    int64_t parts = 0;         // doubles of partials
    int max_log2n = 5;
    size_t o_desc = 0, o_ids = 0, o_tw64 = 0, o_tw32 = 0, o_lap = 0, o_lap32 = 0, o_rho64 = 0,
           o_rho32 = 0, o_fx8 = 0, o_fx4 = 0, o_sc = 0, o_part = 0, o_c32 = 0, o_vec = 0, total = 0;
};

static rve_status make_plan3(const rve_realization* r, int32_t batch, Plan3& p) {
    if (!r || batch <= 0 || batch > (1 << 16)) return RVE_EINVAL;
    p.batch = batch;
    p.desc.assign(2 * (size_t)batch, U3{});
    p.u_of.assign(batch, 0);
    p.nodes = 0;
    p.parts = 0;
    p.max_log2n = 5;
    std::map<int, std::vector<int32_t>> by_size;   // realizations by log2 n
    std::vector<int64_t> cell_off(batch);
    for (int b = 0; b < batch; ++b) {
        const rve_realization& x = r[b];
        if (x.L <= 0 || x.m0 <= 0) return RVE_EINVAL;
        const int64_t n64 = (int64_t)x.L * x.m0;
        if (n64 < N3_MIN || n64 > N3_MAX || (n64 & (n64 - 1))) return RVE_EINVAL;
        const int n = (int)n64;
        if (x.incl_cells <= 0 || x.incl_cells > n || x.n_incl < 0) return RVE_EINVAL;
        if ((int64_t)x.n_incl * x.incl_cells * x.incl_cells > (1LL << 31)) return RVE_EINVAL;
        if (!std::isfinite(x.a_matrix) || !std::isfinite(x.a_incl) || !(x.a_matrix > 0.0) ||
            !(x.a_incl > 0.0))
            return RVE_EINVAL;
        const int lg = 31 - __builtin_clz((unsigned)n);
        by_size[lg].push_back(b);
        cell_off[b] = p.nodes;
        p.nodes += (int64_t)n * n * n;
        p.max_log2n = std::max(p.max_log2n, lg);
    }
    p.unit_nodes = 2 * p.nodes;
    p.groups.clear();
    int u = 0;
    int64_t off = 0;
    for (auto& kv : by_size) {
        Group3 g;
        g.log2n = kv.first;
        g.first = u;
        g.count = 2 * (int)kv.second.size();
        const int half = (int)kv.second.size();
        const int64_t nn = (int64_t)1 << (3 * kv.first);
        for (int pair = 0; pair < 2; ++pair)
            for (int q = 0; q < half; ++q) {
                const int b = kv.second[q];
                const rve_realization& x = r[b];
                U3& d = p.desc[u];
                std::memset(&d, 0, sizeof(d));
                d.n = 1 << kv.first;
                d.log2n = kv.first;
                d.pair = pair;
                d.n_incl = x.n_incl;
                d.s = x.incl_cells;
                d.real = b;
                d.partner = pair == 0 ? g.first + half + q : g.first + q;
                d.cell_off = cell_off[b];
                d.part_off = p.parts;
                d.am = x.a_matrix;
                d.ai = x.a_incl;
                d.am32 = (float)x.a_matrix;
                d.ai32 = (float)x.a_incl;
                d.h = 1.0 / (double)x.m0;
                d.c0 = 0.5 * (x.a_matrix + x.a_incl);
                d.inv_vol = 1.0 / ((double)x.L * (double)x.L * (double)x.L);
                d.key = sm64_mix(x.seed + (x.index + 1) * 0x9E3779B97F4A7C15ull);
                d.off = off;
                if (pair == 0) p.u_of[b] = u;
                off += nn;
                p.parts += A3_NP * (nn / T3);   // enough for every kernel and for A_hom
                ++u;
            }
        p.groups.push_back(g);
    }
    auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
    size_t woff = 0;
    auto take = [&](size_t bytes) { const size_t o = woff; woff = up(woff + bytes); return o; };
    const size_t tab = (size_t)2 << p.max_log2n;
    p.o_desc = take(sizeof(U3) * p.desc.size());
    p.o_ids = take(sizeof(int32_t) * p.u_of.size());
    p.o_tw64 = take(sizeof(double2) * tab);
    p.o_tw32 = take(sizeof(float2) * tab);
    p.o_lap = take(sizeof(double) * tab);
    p.o_lap32 = take(sizeof(float) * tab);
    p.o_rho64 = take(sizeof(double) * tab);
    p.o_rho32 = take(sizeof(float) * tab);
    p.o_fx8 = take(sizeof(int4) * tab);
    p.o_fx4 = take(sizeof(int4) * tab);
    p.o_sc = take(sizeof(MixScal) * p.desc.size());
    p.o_part = take(sizeof(double) * (size_t)p.parts);
    p.o_c32 = take(sizeof(float) * (size_t)p.nodes);
    p.o_vec = take(sizeof(double2) * NVEC * (size_t)p.unit_nodes);
    p.total = woff;
    return RVE_OK;
}

struct Ws3 {   // device pointers into the workspace
    const Plan3* p;
    char* w;
    const U3* desc() const { return reinterpret_cast<const U3*>(w + p->o_desc); }
    const int32_t* u_of() const { return reinterpret_cast<const int32_t*>(w + p->o_ids); }
    MixScal* sc() const { return reinterpret_cast<MixScal*>(w + p->o_sc); }
    double* part() const { return reinterpret_cast<double*>(w + p->o_part); }
    float* c32() const { return reinterpret_cast<float*>(w + p->o_c32); }
    template <typename V> V* vec(int k) const {   // unit vector k, 16 bytes per node reserved
        return reinterpret_cast<V*>(w + p->o_vec + (size_t)k * 16 * (size_t)p->unit_nodes);
    }
    Tables tables() const {
        Tables tb;
        tb.tw64 = reinterpret_cast<const double2*>(w + p->o_tw64);
        tb.tw32 = reinterpret_cast<const float2*>(w + p->o_tw32);
        tb.lap = reinterpret_cast<const double*>(w + p->o_lap);
        tb.lap32 = reinterpret_cast<const float*>(w + p->o_lap32);
        tb.rho64 = reinterpret_cast<const double*>(w + p->o_rho64);
        tb.rho32 = reinterpret_cast<const float*>(w + p->o_rho32);
        tb.fx8 = reinterpret_cast<const int4*>(w + p->o_fx8);
        tb.fx4 = reinterpret_cast<const int4*>(w + p->o_fx4);
        return tb;
    }
    // launch over the units (or the pair-0 units) of group g, `per` (a power
    // of two) blocks each
    Grp grp(const Group3& g, int per, bool reals = false) const {
        (void)reals;   // the pair-0 units come first in the group
        return Grp{desc(), g.first, 31 - __builtin_clz((unsigned)per)};
    }
};
enum { V_F = 0, V_U, V_R64, V_R, V_Z, V_P, V_E, V_Q };

static unsigned nblocks(const Group3& g, int64_t per, bool reals = false) {
    return (unsigned)((reals ? g.count / 2 : g.count) * per);
}
static int64_t nodes_of(const Group3& g) { return (int64_t)1 << (3 * g.log2n); }

// Setup common to the entry points: descriptors, id lists and tables.
static rve_status setup3(const Plan3& p, char* w, cudaStream_t s, bool tables) {
    if (cudaMemcpyAsync(w + p.o_desc, p.desc.data(), sizeof(U3) * p.desc.size(),
                        cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync(w + p.o_ids, p.u_of.data(), sizeof(int32_t) * p.u_of.size(),
                        cudaMemcpyHostToDevice, s) != cudaSuccess)
        return RVE_ECUDA;
    if (!tables) return RVE_OK;
    Ws3 ws{&p, w};
    return fill_tables(ws.tables(), p.max_log2n, s) == cudaSuccess ? RVE_OK : RVE_ECUDA;
}

// The preconditioner's passes over the units of group g, z = M^-1 Hy Hx src / n
// (half 1, with the partials of src.B^-1 src if `rz`), and dst from z (half 2):
// B^-1 src without `e`, the step's new direction and iterate with it.  src is
// read by the first pass only (it may equal z).
template <int LG, typename V>
static cudaError_t precond3_t(const Ws3& ws, const Group3& g, double delta, const V* src, V* z, V* dst,
                              V* e, bool rz, int half, const MixScal* sc, cudaStream_t s) {
    typedef typename ScalarOf<V>::T T;
    constexpr int n = 1 << LG, TL = n / 8;
    const int G = 256 / TL;
    const size_t smem = (size_t)G * seq_stride(n) * sizeof(V);
    const int lines = (n * n) / G;
    constexpr int ZC = zcols<LG>(), ZP = n / ZSEG;
    const size_t zsmem = (size_t)(2 * ZC + 2) * ZP * sizeof(V);
    auto lx = k3_lines<LG, 2, false, V>;
    auto ly = k3_lines<LG, 1, false, V>;
    auto ls = k3_lines<LG, 2, true, V>;
    cudaError_t er = cudaSuccess;
    for (auto k : {lx, ly, ls})
        if (er == cudaSuccess) er = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (er != cudaSuccess) return er;
    const Tables tb = ws.tables();
    const Grp gl = ws.grp(g, lines);
    const unsigned bl = nblocks(g, lines);
    if (half & 1) {
        {
            Span3 sp(s, P3_LINES);
            lx<<<bl, 256, smem, s>>>(gl, tb, src, z, (T)1, nullptr, sc);
        }
        {
            Span3 sp(s, P3_LINES);
            ly<<<bl, 256, smem, s>>>(gl, tb, z, z, (T)1, nullptr, sc);
        }
        {
            Span3 sp(s, P3_ZSOLVE);
            k3_zsolve<LG, V><<<nblocks(g, n * n / ZC), Z_THREADS, zsmem, s>>>(
                ws.grp(g, n * n / ZC), tb, delta, z, rz ? ws.part() : nullptr, sc);
        }
        note_launch(3);
    }
    if (half & 2) {
        {
            Span3 sp(s, P3_LINES);
            ly<<<bl, 256, smem, s>>>(gl, tb, z, z, (T)1, nullptr, sc);
        }
        {
            Span3 sp(s, P3_LINES);
            (e ? ls : lx)<<<bl, 256, smem, s>>>(gl, tb, z, dst, (T)(1.0 / (double)n), e, sc);
        }
        note_launch(2);
    }
    return cudaGetLastError();
}

template <typename V>
static cudaError_t precond3(const Ws3& ws, const Group3& g, double delta, const V* src, V* z, V* dst,
                            V* e, bool rz, int half, const MixScal* sc, cudaStream_t s) {
    switch (g.log2n) {
        case 5: return precond3_t<5, V>(ws, g, delta, src, z, dst, e, rz, half, sc, s);
        case 6: return precond3_t<6, V>(ws, g, delta, src, z, dst, e, rz, half, sc, s);
        case 7: return precond3_t<7, V>(ws, g, delta, src, z, dst, e, rz, half, sc, s);
        default: return precond3_t<8, V>(ws, g, delta, src, z, dst, e, rz, half, sc, s);
    }
}

template <int MODE, typename V>
static cudaError_t stiffness3(const Ws3& ws, const Group3& g, Cells3T<typename ScalarOf<V>::T> cs,
                              int scheme, const V* x, V* y, const V* f, bool partials,
                              const MixScal* sc, cudaStream_t s) {
    const int per = (int)(nodes_of(g) / (2 * T3 * SZ));
    const Grp gg = ws.grp(g, per);
    double* part = partials ? ws.part() : nullptr;
    const size_t smem = stiff_smem<V>(g.log2n);
    auto kern = scheme == RVE_Q1_LUMPED ? k3_stiffness<1, MODE, V> : k3_stiffness<0, MODE, V>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    Span3 sp(s, MODE == MODE_RESID ? P3_RESID : P3_STIFF);
    kern<<<nblocks(g, per), T3, smem, s>>>(gg, cs, x, y, f, part, sc);
    note_launch();
    return cudaGetLastError();
}

// r64 = f - A u of the units of group g in double words (the mixed path):
// u split into double words in the q slot, then the residual pass.
static cudaError_t resid3_dw(const Ws3& ws, const Group3& g, Cells3T<double> cs, int scheme,
                             const double2* u, double2* r, const double2* f, const MixScal* sc,
                             cudaStream_t s) {
    const int per = (int)(nodes_of(g) / T3);
    float4* wdw = reinterpret_cast<float4*>(ws.vec<double2>(V_Q));   // 16 bytes per node
    const Grp gg = ws.grp(g, per);
    Span3 sp(s, P3_RESID);
    k3_split_dw<<<nblocks(g, per), T3, 0, s>>>(gg, u, wdw, ws.sc());
    if (scheme == RVE_Q1_LUMPED)
        k3_resid_dw<1><<<nblocks(g, per), T3, 0, s>>>(gg, cs, wdw, f, r, ws.part(), sc);
    else
        k3_resid_dw<0><<<nblocks(g, per), T3, 0, s>>>(gg, cs, wdw, f, r, ws.part(), sc);
    note_launch(2);
    return cudaGetLastError();
}

// The correctors of every unit: cycles of PCG in the precision of V between
// FP64 true residuals (see the head of the file).
template <typename V>
static rve_status solve_units(const Plan3& p, char* w, Cells3T<double> cs64,
                              Cells3T<typename ScalarOf<V>::T> csV, const rve3_solve_opts& o,
                              cudaStream_t s) {
    const Ws3 ws{&p, w};
    MixScal* sc = ws.sc();
    double* part = ws.part();
    double2* f = ws.vec<double2>(V_F);
    double2* uv = ws.vec<double2>(V_U);
    double2* r64 = ws.vec<double2>(V_R64);
    V* r = ws.vec<V>(V_R);
    V* z = ws.vec<V>(V_Z);
    V* pp = ws.vec<V>(V_P);
    V* e = ws.vec<V>(V_E);
    V* q = ws.vec<V>(V_Q);
    const bool fp64 = sizeof(typename ScalarOf<V>::T) == 8;
    const ScalArgs sa{o.tol, fp64 ? 0.0 : o.inner_tol, fp64 ? 1.0 : 0.5, o.max_iter};
    auto vec_step = [&](auto&& launch) {
        Span3 sp(s, P3_VECTOR);
        launch();
    };
    // partial pairs per unit: n^3 >> shift (rhs: 256 nodes per block; update:
    // 1024; stiffness: 2048; z solve: 8192)
    constexpr int SH_RHS = 8, SH_STIFF = 11, SH_AXPY = 10, SH_Z = 13;
    static_assert(2 * T3 * SZ == (1 << SH_STIFF) && 4 * T3 == (1 << SH_AXPY) && T3 == (1 << SH_RHS) &&
                      Z_THREADS * ZSEG == (1 << SH_Z),
                  "partial counts");
    auto scalar = [&](const Group3& g, int what, int shift) {
        Span3 sp(s, P3_SCALAR);
        k3_scalar<<<g.count, 256, 0, s>>>(g.first, ws.desc(), sc, part, what, shift, sa);
        note_launch();
    };
    // z = B^-1 r with r.z, then the scalar step, then e += alpha p, p = z + beta p
    auto direction = [&](const Group3& g, int what) -> bool {
        if (precond3<V>(ws, g, o.delta, r, z, pp, e, true, 1, sc, s) != cudaSuccess) return false;
        scalar(g, what, SH_Z);
        return precond3<V>(ws, g, o.delta, r, z, pp, e, true, 2, sc, s) == cudaSuccess;
    };
    auto per_group = [&](auto&& fn) -> rve_status {
        for (const Group3& g : p.groups) {
            const rve_status st = fn(g);
            if (st != RVE_OK) return st;
        }
        return cudaGetLastError() == cudaSuccess ? RVE_OK : RVE_ECUDA;
    };
    std::vector<MixScal> hsc(p.desc.size());
    auto poll = [&](bool outer) -> int {   // -1 error, 1 every unit finished
        if (cudaMemcpyAsync(hsc.data(), sc, sizeof(MixScal) * hsc.size(), cudaMemcpyDeviceToHost, s) !=
                cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return -1;
        if (profile_on()) g_prof3.harvest();
        for (const MixScal& m : hsc)
            if (!(outer ? m.outer_done : m.done)) return 0;
        return 1;
    };
    rve_status st;
    // loads with |f|^2, u = 0
    st = per_group([&](const Group3& g) {
        const int per = (int)(nodes_of(g) / T3);
        vec_step([&] { k3_rhs<<<nblocks(g, per), T3, 0, s>>>(ws.grp(g, per), cs64, f, part); });
        scalar(g, M_FNORM, SH_RHS);
        note_launch();
        return RVE_OK;
    });
    if (st != RVE_OK) return st;
    if (cudaMemsetAsync(uv, 0, sizeof(double2) * (size_t)p.unit_nodes, s) != cudaSuccess ||
        cudaMemcpyAsync(r64, f, sizeof(double2) * (size_t)p.unit_nodes, cudaMemcpyDeviceToDevice, s) !=
            cudaSuccess)
        return RVE_ECUDA;
    const int every = o.check_every;
    for (int cycle = 0; cycle <= MAX_REFINE + 1; ++cycle) {
        // FP64 true residual r64 = f - A u and the refinement step
        st = per_group([&](const Group3& g) {
            int shift = SH_RHS;   // u = 0: r64 = f, the partials of |f|^2 are still in place
            if (cycle > 0 && fp64) {
                if (stiffness3<MODE_RESID, double2>(ws, g, cs64, o.scheme, uv, r64, f, true, sc, s) !=
                    cudaSuccess)
                    return RVE_ECUDA;
                shift = SH_STIFF;
            } else if (cycle > 0) {   // mixed: the double-word residual
                if (resid3_dw(ws, g, cs64, o.scheme, uv, r64, f, sc, s) != cudaSuccess)
                    return RVE_ECUDA;
                shift = SH_RHS;
            }
            scalar(g, M_REFINE, shift);
            return RVE_OK;
        });
        if (st != RVE_OK) return st;
        const int pr = poll(true);
        if (pr < 0) return RVE_ECUDA;
        if (pr == 1) break;
        // a cycle: r = r64 / s, z = B^-1 r, p = z
        st = per_group([&](const Group3& g) {
            const int per = (int)(nodes_of(g) / T3);
            vec_step([&] { k3_start<V><<<nblocks(g, per), T3, 0, s>>>(ws.grp(g, per), sc, r64, r, e, pp); });
            note_launch();
            return direction(g, M_RHO0) ? RVE_OK : RVE_ECUDA;   // alpha = beta = 0, e = p = 0
        });
        if (st != RVE_OK) return st;
        for (int it = 1;; ++it) {
            st = per_group([&](const Group3& g) {
                const int per = (int)(nodes_of(g) / T3), per4 = per / 4;
                if (stiffness3<MODE_APPLY, V>(ws, g, csV, o.scheme, pp, q, nullptr, true, sc, s) !=
                    cudaSuccess)
                    return RVE_ECUDA;
                scalar(g, M_ALPHA, SH_STIFF);
                vec_step([&] {
                    k3_update<V><<<nblocks(g, per4), T3, 0, s>>>(ws.grp(g, per4), sc, r, q, part);
                });
                scalar(g, M_CONV, SH_AXPY);
                note_launch();
                return direction(g, M_BETA) ? RVE_OK : RVE_ECUDA;
            });
            if (st != RVE_OK) return st;
            if (it % every == 0) {
                const int pi = poll(false);
                if (pi < 0) return RVE_ECUDA;
                if (pi == 1) break;
            }
        }
        st = per_group([&](const Group3& g) {
            const int per = (int)(nodes_of(g) / T3);
            vec_step([&] { k3_accum<V><<<nblocks(g, per), T3, 0, s>>>(ws.grp(g, per), sc, e, pp, uv); });
            note_launch();
            return RVE_OK;
        });
        if (st != RVE_OK) return st;
    }
    return RVE_OK;
}

static rve3_solve_opts resolved3(const rve3_solve_opts* opts) {
    rve3_solve_opts o = {};
    if (opts) o = *opts;
    if (o.max_iter <= 0) o.max_iter = 20000;
    if (!(o.tol > 0.0)) o.tol = 1e-10;
    if (!(o.inner_tol > 0.0)) o.inner_tol = 1e-4;
    if (o.check_every <= 0) o.check_every = 8;
    return o;
}

static bool valid_scheme(int s) { return s == RVE_Q1_CONSISTENT || s == RVE_Q1_LUMPED; }

}  // namespace rve

using namespace rve;

extern "C" {

int64_t rve3_nodes(const rve_realization* r, int32_t batch) {
    Plan3 p;
    return make_plan3(r, batch, p) == RVE_OK ? p.nodes : -1;
}

size_t rve3_workspace_size(const rve_realization* r, int32_t batch) {
    Plan3 p;
    return make_plan3(r, batch, p) == RVE_OK ? p.total : 0;
}

rve_status rve3_gen_field(const rve_realization* r, int32_t batch, uint8_t* mask, void* stream) {
    Plan3 p;
    rve_status st = make_plan3(r, batch, p);
    if (st != RVE_OK) return st;
    if (!mask) return RVE_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(mask, 0, (size_t)p.nodes, s) != cudaSuccess) return RVE_ECUDA;
    for (int b = 0; b < p.batch; ++b) {
        const U3& d = p.desc[p.u_of[b]];
        const int64_t rows = (int64_t)d.n_incl * d.s * d.s;
        if (rows == 0) continue;
        k3_gen_field<<<(unsigned)((rows + 255) / 256), 256, 0, s>>>(d, mask);
        note_launch();
    }
    return cudaGetLastError() == cudaSuccess ? RVE_OK : RVE_ECUDA;
}

rve_status rve3_rhs(const rve_realization* r, int32_t batch, const uint8_t* mask, const double* coef,
                    int32_t scheme, double* f, void* ws, size_t ws_bytes, void* stream) {
    Plan3 p;
    rve_status st = make_plan3(r, batch, p);
    if (st != RVE_OK) return st;
    if ((!mask && !coef) || !f || !ws || ws_misaligned(ws) || !valid_scheme(scheme)) return RVE_EINVAL;
    if (ws_bytes < p.total) return RVE_ENOMEM;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    char* w = static_cast<char*>(ws);
    if ((st = setup3(p, w, s, false)) != RVE_OK) return st;
    const Ws3 W{&p, w};
    const Cells3T<double> cs{mask, coef};
    for (const Group3& g : p.groups) {
        const int per = (int)(nodes_of(g) / T3);
        k3_rhs<<<nblocks(g, per), T3, 0, s>>>(W.grp(g, per), cs, W.vec<double2>(V_F), nullptr);
        k3_join<<<nblocks(g, per), T3, 0, s>>>(W.grp(g, per), W.vec<double2>(V_F), f);
        note_launch(2);
    }
    return cudaGetLastError() == cudaSuccess ? RVE_OK : RVE_ECUDA;
}

rve_status rve3_apply_stiffness(const rve_realization* r, int32_t batch, const uint8_t* mask,
                                const double* coef, int32_t scheme, const double* x, double* y,
                                void* ws, size_t ws_bytes, void* stream) {
    Plan3 p;
    rve_status st = make_plan3(r, batch, p);
    if (st != RVE_OK) return st;
    if ((!mask && !coef) || !x || !y || x == y || !ws || ws_misaligned(ws) || !valid_scheme(scheme))
        return RVE_EINVAL;
    if (ws_bytes < p.total) return RVE_ENOMEM;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    char* w = static_cast<char*>(ws);
    if ((st = setup3(p, w, s, false)) != RVE_OK) return st;
    const Ws3 W{&p, w};
    const Cells3T<double> cs{mask, coef};
    for (const Group3& g : p.groups) {
        const int per = (int)(nodes_of(g) / T3);
        k3_split<<<nblocks(g, per), T3, 0, s>>>(W.grp(g, per), x, W.vec<double2>(V_R));
        note_launch();
        if (stiffness3<MODE_APPLY, double2>(W, g, cs, scheme, W.vec<double2>(V_R), W.vec<double2>(V_Q),
                                            nullptr, false, nullptr, s) != cudaSuccess)
            return RVE_ECUDA;
        k3_join<<<nblocks(g, per), T3, 0, s>>>(W.grp(g, per), W.vec<double2>(V_Q), y);
        note_launch();
    }
    return cudaGetLastError() == cudaSuccess ? RVE_OK : RVE_ECUDA;
}

rve_status rve3_apply_precond(const rve_realization* r, int32_t batch, double delta,
                              const double* x, double* y, void* ws, size_t ws_bytes,
                              void* stream) {
    Plan3 p;
    rve_status st = make_plan3(r, batch, p);
    if (st != RVE_OK) return st;
    if (!x || !y || !ws || ws_misaligned(ws) || !std::isfinite(delta) || delta < 0.0) return RVE_EINVAL;
    if (ws_bytes < p.total) return RVE_ENOMEM;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    char* w = static_cast<char*>(ws);
    if ((st = setup3(p, w, s, true)) != RVE_OK) return st;
    const Ws3 W{&p, w};
    double2* v = W.vec<double2>(V_R);
    for (const Group3& g : p.groups) {
        const int per = (int)(nodes_of(g) / T3);
        k3_split<<<nblocks(g, per), T3, 0, s>>>(W.grp(g, per), x, v);
        note_launch();
    }
    for (const Group3& g : p.groups)
        if (precond3<double2>(W, g, delta, v, v, v, nullptr, false, 3, nullptr, s) != cudaSuccess) return RVE_ECUDA;
    for (const Group3& g : p.groups) {
        const int per = (int)(nodes_of(g) / T3);
        k3_join<<<nblocks(g, per), T3, 0, s>>>(W.grp(g, per), v, y);
        note_launch();
    }
    return cudaGetLastError() == cudaSuccess ? RVE_OK : RVE_ECUDA;
}

rve_status rve3_solve_correctors(const rve_realization* r, int32_t batch, const uint8_t* mask,
                                 const double* coef, const rve3_solve_opts* opts, double* u,
                                 rve3_solve_info* info, void* ws, size_t ws_bytes,
                                 void* stream) {
    const rve3_solve_opts o = resolved3(opts);
    if (!valid_scheme(o.scheme)) return RVE_EINVAL;
    if (o.precision != RVE_FP64 && o.precision != RVE_MIXED) return RVE_EINVAL;
    if (!std::isfinite(o.delta) || o.delta < 0.0 || !(o.tol < 1.0) || !(o.inner_tol < 1.0))
        return RVE_EINVAL;
    Plan3 p;
    rve_status st = make_plan3(r, batch, p);
    if (st != RVE_OK) return st;
    if ((!mask && !coef) || !u || !info || !ws || ws_misaligned(ws)) return RVE_EINVAL;
    if (ws_bytes < p.total) return RVE_ENOMEM;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    char* w = static_cast<char*>(ws);
    if ((st = setup3(p, w, s, true)) != RVE_OK) return st;
    const Ws3 W{&p, w};
    const Cells3T<double> cs64{mask, coef};
    if (o.precision == RVE_MIXED) {
        if (coef) {
            k3_coef32<<<(unsigned)((p.nodes + 255) / 256), 256, 0, s>>>(coef, W.c32(), p.nodes);
            note_launch();
        }
        const Cells3T<float> cs32{mask, coef ? W.c32() : nullptr};
        st = solve_units<float2>(p, w, cs64, cs32, o, s);
    } else {
        st = solve_units<double2>(p, w, cs64, cs64, o, s);
    }
    if (st != RVE_OK) return st;
    for (const Group3& g : p.groups) {
        const int per = (int)(nodes_of(g) / T3);
        k3_join<<<nblocks(g, per), T3, 0, s>>>(W.grp(g, per), W.vec<double2>(V_U), u);
        note_launch();
    }
    k3_report<<<(p.batch + 127) / 128, 128, 0, s>>>(W.sc(), W.desc(), W.u_of(), p.batch, info);
    note_launch();
    if (cudaGetLastError() != cudaSuccess) return RVE_ECUDA;
    prof3_sync(s);
    return RVE_OK;
}

rve_status rve3_a_hom(const rve_realization* r, int32_t batch, const uint8_t* mask,
                      const double* coef, int32_t scheme, const double* u, double* A,
                      double* A_flux, void* ws, size_t ws_bytes, void* stream) {
    Plan3 p;
    rve_status st = make_plan3(r, batch, p);
    if (st != RVE_OK) return st;
    if ((!mask && !coef) || !u || !A || !ws || ws_misaligned(ws) || !valid_scheme(scheme)) return RVE_EINVAL;
    if (ws_bytes < p.total) return RVE_ENOMEM;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    char* w = static_cast<char*>(ws);
    if ((st = setup3(p, w, s, false)) != RVE_OK) return st;
    const Ws3 W{&p, w};
    const Cells3T<double> cs{mask, coef};
    for (const Group3& g : p.groups) {
        const int per = (int)(nodes_of(g) / T3);
        const int tiles = per / A3_PLANES;
        const Grp gr = W.grp(g, tiles, true);
        if (scheme == RVE_Q1_LUMPED)
            k3_a_hom_part<1><<<nblocks(g, tiles, true), T3, 0, s>>>(gr, cs, u, W.part());
        else
            k3_a_hom_part<0><<<nblocks(g, tiles, true), T3, 0, s>>>(gr, cs, u, W.part());
        k3_a_hom_final<<<g.count / 2, 32 * A3_NP, 0, s>>>(W.grp(g, 1, true), W.part(), A, A_flux);
        note_launch(2);
    }
    return cudaGetLastError() == cudaSuccess ? RVE_OK : RVE_ECUDA;
}

rve_status rve3_statistics(const double* A, int64_t N, double L, double* mean, double* var,
                           double* Q) {
    if (!A || N < 2 || !(L > 0.0) || !std::isfinite(L)) return RVE_EINVAL;
    double m[9] = {};
    for (int64_t k = 0; k < N; ++k)
        for (int e = 0; e < 9; ++e) m[e] += A[9 * k + e];
    for (int e = 0; e < 9; ++e) m[e] /= (double)N;
    std::vector<double> c(81, 0.0);
    for (int64_t k = 0; k < N; ++k) {
        double dev[9];
        for (int e = 0; e < 9; ++e) dev[e] = A[9 * k + e] - m[e];
        for (int i = 0; i < 9; ++i)
            for (int j = 0; j < 9; ++j) c[9 * i + j] += dev[i] * dev[j];
    }
    const double L3 = L * L * L;
    for (int e = 0; e < 9; ++e) {
        if (mean) mean[e] = m[e];
        if (var) var[e] = c[10 * e] / (double)(N - 1);
    }
    if (Q)
        for (int e = 0; e < 81; ++e) Q[e] = L3 * c[e] / (double)(N - 1);
    return RVE_OK;
}

int32_t rve3_profile_read(double* ms, int64_t* launches) {
    for (int j = 0; j < P3_K; ++j) {
        if (ms) ms[j] = g_prof3.ms[j];
        if (launches) launches[j] = (int64_t)g_prof3.launches[j];
        g_prof3.ms[j] = 0.0;
        g_prof3.launches[j] = 0;
    }
    return P3_K;
}

}  // extern "C"
