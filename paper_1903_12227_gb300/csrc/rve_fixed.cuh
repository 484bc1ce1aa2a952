// rve_fixed.cuh -- the row transforms of double pairs in 64-bit fixed point.
//
// GB300 issues 2 FP64 operations per clock and SM but 64 integer ones, and a
// Stockham transform of n = 512 costs 34 FP64 operations per node: the row
// transforms were 55 to 75 % of every FP64 pass.  A Fourier transform mixes
// all elements of its row, so its error is relative to the row's norm in any
// arithmetic; a row scaled by one common power of two and carried in 64-bit
// integers therefore loses nothing against FP64: additions are exact,
// products are rounded at the last of 58 or more bits.
//
// Format.  A row's elements become integers x 2^(FX_BITS - E), E the largest
// exponent of the row, so every component is below 2^58 and every modulus
// below 2^58.5.  The twiddles in front of a stage carry a factor 1/8 or 1/4,
// chosen so that moduli stay below 2^61.5 after every stage (a stage's outputs
// are sums of at most 8^stage elements, and never more than the row's 1-norm);
// the Hartley sum of four components of the last stage then stays below 2^63.
// With c the row's 1-norm over 2^58.5 the schedule is (fx_schedule):
//   in front of stage 2: 1/8, or 1/4 for c <= 32;
//   in front of stage 3 (radix 8): 1/8, or 1/4 for c <= 256;
//   in front of a radix-4 or radix-2 tail: 1/4.
// Dense rows (c about n/4) need every bit of head room; rows of few large
// elements (spectra) do not, and the unit they lose least by is a finer one.
//
// Error of one row (2-norm, against long double, as a part of that of the same
// stages in double; tests/fixed_rows_host.cu): noise, smooth and dense rows 0.32 to
// 0.72; spikes, heavy tails and spectra at most 0.65 up to n = 512, 0.94 at 1024,
// 1.08 at 2048.  The worst rows found, a spike on noise of 1 to 5 % of it, reach
// 1.4 and 1.5 at 1024 and 2048: three divisions where the row hardly grows.  (Giving
// those bits back behind each product brings every row to 0.70 or less, and costs
// a 1024^2 FP64 solve 2.6 %.)  Error of a whole B^-1 x (two row transforms and the
// column pass, against 128-bit FFTs; noise, spikes, a spike on noise, smooth fields
// and corrector loads, 512^2 to 2048^2): 0.75 to 0.99 of the FP64 form's.
// Rows with an infinity or a NaN, rows so large that a result could overflow,
// and rows so small that one could be subnormal, take the FP64 transform
// (fx_takes).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace rve {

typedef long long fx_t;
constexpr int FX_BITS = 57;       // the row's largest component is in [2^57, 2^58)
// Biased exponents taken.  A component of the result has at most 13 more than
// the row's largest (2048 elements of modulus below 2^1.5 times its binade, and
// the rounding), and a double's largest is 2046.
constexpr unsigned FX_E_MIN = 128, FX_E_MAX = 2046 - 13;

// High and low word of v, the low one signed (v = h 2^32 + l).
__host__ __device__ __forceinline__ void fx_split(fx_t v, int& h, int& l) {
    l = (int)(uint32_t)(uint64_t)v;
    h = (int)((v + 0x80000000ll) >> 32);
}
// Twiddle (cos, sin) / 2^lr as 64-bit fractions (c.h, c.l, s.h, s.l), lr = 3
// or 2; low words kept above -2^31 so that they can be negated.
__host__ __device__ __forceinline__ int4 fx_twiddle(double c, double s, int lr) {
    int4 w;
    const double k = lr == 3 ? 2305843009213693952.0 : 4611686018427387904.0;   // 2^(64 - lr)
    fx_split((fx_t)(c * k), w.x, w.y);
    fx_split((fx_t)(s * k), w.z, w.w);
    if (w.y == INT32_MIN) w.y += 1;
    if (w.w == INT32_MIN) w.w += 1;
    return w;
}
__host__ __device__ __forceinline__ fx_t fx_wide(int a, int b) { return (fx_t)a * (fx_t)b; }

// a times the twiddle w for |a| < 2^61.5: the products of the high words, and
// those of the mixed words (their sums stay below 2^63) rounded at 2^32; low
// times low is below half a unit.
__host__ __device__ __forceinline__ longlong2 cmul(longlong2 a, int4 w) {
    int rh, rl, ih, il;
    fx_split(a.x, rh, rl);
    fx_split(a.y, ih, il);
    const int nsh = -w.z, nsl = -w.w;
    const fx_t half = 1ll << 31;
    const fx_t cr = half + fx_wide(rh, w.y) + fx_wide(rl, w.x) + fx_wide(ih, nsl) + fx_wide(il, nsh);
    const fx_t ci = half + fx_wide(rh, w.w) + fx_wide(rl, w.z) + fx_wide(ih, w.y) + fx_wide(il, w.x);
    longlong2 r;
    r.x = (cr >> 32) + fx_wide(rh, w.x) + fx_wide(ih, nsh);
    r.y = (ci >> 32) + fx_wide(rh, w.z) + fx_wide(ih, w.x);
    return r;
}
// The element that takes no twiddle: a / 2^k, rounded.
__host__ __device__ __forceinline__ longlong2 fx_shift(longlong2 a, int k) {
    const fx_t half = 1ll << (k - 1);
    longlong2 r;
    r.x = (a.x + half) >> k;
    r.y = (a.y + half) >> k;
    return r;
}
// v / sqrt(2) = v - v (1 - 1/sqrt(2)).
__host__ __device__ __forceinline__ fx_t fx_rsqrt2(fx_t v) {
    constexpr fx_t k = 5402926248376769404ll;   // (1 - 2^-1/2) 2^64, rounded
    constexpr int kl = (int)(uint32_t)(uint64_t)k, kh = (int)((k + 0x80000000ll) >> 32);
    int h, l;
    fx_split(v, h, l);
    const fx_t c = (1ll << 31) + fx_wide(h, kl) + fx_wide(l, kh);
    return v - (fx_wide(h, kh) + (c >> 32));
}

// double x -> round(x 2^(FX_BITS - (E - 1023))), E >= the biased exponent of x.
__host__ __device__ __forceinline__ fx_t fx_from(double x, unsigned E) {
#ifdef __CUDA_ARCH__
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
#else
    union { double d; uint64_t u; } c;
    c.d = x;
    const unsigned hi = (unsigned)(c.u >> 32), lo = (unsigned)c.u;
#endif
    const unsigned e = (hi >> 20) & 0x7FFu;
    // the 53-bit significand with its leading bit at 2^63; subnormals are far
    // below the unit
    const uint64_t m = ((uint64_t)(0x80000000u | ((hi & 0xFFFFFu) << 11) | (lo >> 21)) << 32) |
                       (uint64_t)(lo << 11);
    // keep one bit below the unit for the rounding
    const unsigned sh = (63 - FX_BITS - 1) + (E - e);
    const uint64_t t = (sh > 63u || e == 0u) ? 0ull : (m >> sh);
    const fx_t v = (fx_t)((t + 1) >> 1);
    return (hi >> 31) ? -v : v;
}

// The double v 2^(q - 1023), rounded to nearest (q + 63 in the normal range).
__host__ __device__ __forceinline__ double fx_to(fx_t v, int q) {
    const uint64_t s = (uint64_t)(v >> 63);
    uint64_t u = ((uint64_t)v ^ s) - s;
#ifdef __CUDA_ARCH__
    const int lz = __clzll((long long)u);
#else
    const int lz = u ? __builtin_clzll(u) : 64;
#endif
    u <<= (lz & 63);
    const uint64_t m = (u >> 11) + ((u >> 10) & 1);   // 2^52 <= m <= 2^53
    const uint64_t bits = ((uint64_t)(unsigned)(q + 62 - lz) << 52) + m;
    const uint64_t r = (v == 0) ? 0ull : (bits | (s << 63));
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)r);
#else
    union { double d; uint64_t u; } c;
    c.u = r;
    return c.d;
#endif
}

// High word of a component without its sign, 1 where only the low word is set
// (0: the component is zero).
__host__ __device__ __forceinline__ unsigned fx_high(unsigned hi, unsigned lo) {
    hi &= 0x7FFFFFFFu;
    return hi != 0u ? hi : (unsigned)(lo != 0u);
}
// Biased exponent of a row whose largest fx_high is `hi`.  A row of zeros fits any
// unit (in FP64 it was slower, and so were the rows that shared its warp: 1000 x
// 64^2 nodes, every third row zero, 554 us, with none 405, now 403).
__host__ __device__ __forceinline__ unsigned fx_row_exponent(unsigned hi) { return hi == 0u ? 1023u : hi >> 20; }
// A row's largest biased exponent is in range.
__host__ __device__ __forceinline__ bool fx_takes(unsigned E) { return E >= FX_E_MIN && E <= FX_E_MAX; }
// Size of a component with high word `hi`, in units of 2^40 (rounded down;
// the largest of the row has 2^17 to 2^18): its row's 1-norm is below 2^40
// (sum of the sizes + 2 n).
__host__ __device__ __forceinline__ unsigned fx_size(unsigned hi, unsigned E) {
    const unsigned e = (hi >> 20) & 0x7FFu;
    return (0x20000u | ((hi & 0xFFFFFu) >> 3)) >> (E - e < 31u ? E - e : 31u);
}
// Halvings in front of stages 2, 3 and 4 (a tail's are fixed) of a row of 2^p
// pairs; `sum`: of its sizes (only looked at from p = 7 on: below, a spike
// costs no accuracy at the widest schedule).  `finer`: the unit may be halved
// (c <= 4: nothing ever exceeds the 1-norm).
struct FxShifts { int s2, s3, s4; unsigned finer; };
__host__ __device__ __forceinline__ FxShifts fx_schedule(int p, unsigned sum) {
    const unsigned one = 370727u;   // 2^58.5 in units of 2^40
    const unsigned norm = sum + (2u << p);
    FxShifts f;
    f.s2 = (p == 5 || (p >= 7 && norm <= 32u * one)) ? 2 : 3;
    f.s3 = (p < 9 || norm <= 256u * one) ? 2 : 3;
    f.s4 = 2;
    f.finer = (p >= 7 && norm <= 4u * one) ? 1u : 0u;
    return f;
}
__host__ __device__ __forceinline__ int fx_scale(int p, const FxShifts& f) {
    return f.s2 + (p > 6 ? f.s3 : 0) + (p > 9 ? f.s4 : 0);
}

}  // namespace rve
