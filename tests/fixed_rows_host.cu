// Host run of the fixed-point row transform (csrc/rve_fixed.cuh): the stages
// of fft_reg with its arithmetic, every intermediate checked against its bound
// in 128 bits, and the error against a long double DFT beside that of the same
// stages in double.  Prints "p kind fixed_error double_error" per row set.
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <vector>

#include "rve_fixed.cuh"
using namespace rve;

typedef longlong2 L2;
typedef std::complex<double> C;

static void within(__int128 v, int bits) {
    if ((v < 0 ? -v : v) >> bits) {
        std::printf("a value exceeds 2^%d\n", bits);
        std::exit(1);
    }
}
static L2 add(L2 a, L2 b) { within((__int128)a.x + b.x, 63); within((__int128)a.y + b.y, 63); return L2{a.x + b.x, a.y + b.y}; }
static L2 sub(L2 a, L2 b) { within((__int128)a.x - b.x, 63); within((__int128)a.y - b.y, 63); return L2{a.x - b.x, a.y - b.y}; }
static C add(C a, C b) { return a + b; }
static C sub(C a, C b) { return a - b; }
static L2 mi(L2 a) { return L2{a.y, -a.x}; }
static C mi(C a) { return C(a.imag(), -a.real()); }
static L2 rot(L2 a, int s) {   // times exp(-i pi s / 4), s = 1 or 3
    within((__int128)a.x + a.y, 63);
    within((__int128)a.y - a.x, 63);
    return s == 1 ? L2{fx_rsqrt2(a.x + a.y), fx_rsqrt2(a.y - a.x)}
                  : L2{fx_rsqrt2(a.y - a.x), -fx_rsqrt2(a.x + a.y)};
}
static C rot(C a, int s) {
    const double c = std::sqrt(0.5);
    return s == 1 ? C(c * (a.real() + a.imag()), c * (a.imag() - a.real()))
                  : C(c * (a.imag() - a.real()), -c * (a.real() + a.imag()));
}
static L2 times(L2 a, double c, double s, int k) {
    within(a.x, 62);
    within(a.y, 62);
    const int4 w = fx_twiddle(c, s, k);
    int rh, rl, ih, il;
    fx_split(a.x, rh, rl);
    fx_split(a.y, ih, il);
    const __int128 half = (__int128)1 << 31;
    within(half + (__int128)rh * w.y + (__int128)rl * w.x - (__int128)ih * w.w - (__int128)il * w.z, 63);
    within(half + (__int128)rh * w.w + (__int128)rl * w.z + (__int128)ih * w.y + (__int128)il * w.x, 63);
    return cmul(a, w);
}
static C times(C a, double c, double s, int) {
    return C(std::fma(a.real(), c, -(a.imag() * s)), std::fma(a.real(), s, a.imag() * c));
}
static L2 shift(L2 a, int k) { return fx_shift(a, k); }
static C shift(C a, int) { return a; }

template <typename V> static void d4(V& a, V& b, V& c, V& d) {
    const V s = add(a, c), e = sub(a, c), t = add(b, d), f = mi(sub(b, d));
    a = add(s, t); c = sub(s, t); b = add(e, f); d = sub(e, f);
}
template <typename V> static void d8(V* u) {
    V e[4] = {u[0], u[2], u[4], u[6]}, o[4] = {u[1], u[3], u[5], u[7]};
    d4(e[0], e[1], e[2], e[3]);
    d4(o[0], o[1], o[2], o[3]);
    const V t[4] = {o[0], rot(o[1], 1), mi(o[2]), rot(o[3], 3)};
    for (int k = 0; k < 4; ++k) { u[k] = add(e[k], t[k]); u[k + 4] = sub(e[k], t[k]); }
}
template <typename V> static void fft(std::vector<V>& x, int p, const FxShifts& f) {
    const int n = 1 << p;
    std::vector<V> y(n);
    for (int done = 0, stage = 0; done < p; ++stage) {
        const int lr = p - done < 3 ? p - done : 3, R = 1 << lr, Ns = 1 << done, step = n >> lr;
        const int k2 = stage == 1 ? f.s2 : stage == 2 ? f.s3 : f.s4;
        for (int j = 0; j < step; ++j) {
            const int k = j & (Ns - 1);
            V v[8];
            for (int r = 0; r < R; ++r) {
                v[r] = x[j + r * step];
                if (Ns == 1) continue;
                const double a = 2.0 * (double)(r * k) / (double)(Ns * R);
                v[r] = r == 0 ? shift(v[r], k2)
                              : times(v[r], (double)cosl(M_PIl * a), (double)-sinl(M_PIl * a), k2);
            }
            if (R == 8) d8(v);
            else if (R == 4) d4(v[0], v[1], v[2], v[3]);
            else { const V t = v[0]; v[0] = add(t, v[1]); v[1] = sub(t, v[1]); }
            for (int r = 0; r < R; ++r) y[((j - k) << lr) + k + r * Ns] = v[r];
        }
        x.swap(y);
        done += lr;
    }
}
static unsigned high(double x) { uint64_t u; std::memcpy(&u, &x, 8); return (unsigned)(u >> 32); }

int main() {
    std::mt19937_64 g(1);
    std::normal_distribution<double> N(0, 1);
    const double top = std::nextafter(2.0, 0.0);
    for (int p = 5; p <= 11; ++p) {
        const int n = 1 << p;
        std::vector<long double> cas(n);
        for (int m = 0; m < n; ++m) cas[m] = cosl(2 * M_PIl * m / n) + sinl(2 * M_PIl * m / n);
        for (int kind = 0; kind < 9; ++kind) {
            long double ef = 0, ed = 0, norm = 0;
            for (int rep = 0; rep < (n > 512 ? 2 : 5); ++rep) {
                std::vector<double> a(n), b(n);
                for (int i = 0; i < n; ++i) {
                    const double th = 2 * M_PI * i / n, k = std::min(i, n - i);
                    switch (kind) {
                        case 0: a[i] = N(g); b[i] = N(g); break;                               // noise
                        case 1: a[i] = sin(th) + 0.3 * cos(3 * th + rep); b[i] = 1e-3 * cos(2 * th); break;
                        case 2: a[i] = i == 3 * rep; b[i] = i == 5; break;                     // spikes
                        case 3: a[i] = top; b[i] = (rep & 1) ? -top : top; break;              // the bounds
                        case 4: a[i] = (i & 1) ? -top : top; b[i] = (i & 2) ? -top : top; break;
                        case 5: a[i] = N(g) * exp(3 * N(g)); b[i] = 1e-6 * N(g); break;        // heavy tails
                        case 6: a[i] = cos((7 * rep + 3) * th) >= 0 ? top : -top;
                                b[i] = sin((7 * rep + 3) * th) >= 0 ? top : -top; break;
                        case 7: a[i] = N(g) / (1e-4 * n + k * k); b[i] = N(g) / (1 + k); break;   // a spectrum
                        default: a[i] = i < 2 + rep ? top : 0; b[i] = i < 2 ? -top : 0;
                    }
                }
                unsigned E = 0, size = 0;
                for (int i = 0; i < n; ++i)
                    E = std::max(E, std::max((high(a[i]) >> 20) & 0x7FFu, (high(b[i]) >> 20) & 0x7FFu));
                for (int i = 0; i < n; ++i) size += fx_size(high(a[i]), E) + fx_size(high(b[i]), E);
                const FxShifts f = fx_schedule(p, size);
                E -= f.finer;
                std::vector<L2> x(n);
                std::vector<C> z(n);
                for (int i = 0; i < n; ++i) {
                    x[i] = L2{fx_from(a[i], E), fx_from(b[i], E)};
                    z[i] = C(a[i], b[i]);
                }
                fft(x, p, f);
                fft(z, p, f);
                const int q = (int)E - FX_BITS + fx_scale(p, f) - 1;
                for (int k = 0; k < n; ++k) {
                    const int m = (n - k) & (n - 1);
                    const __int128 hx = ((__int128)x[k].x + x[m].x) - ((__int128)x[k].y - x[m].y);
                    const __int128 hy = ((__int128)x[k].y + x[m].y) + ((__int128)x[k].x - x[m].x);
                    within(hx, 63);
                    within(hy, 63);
                    long double ra = 0, rb = 0;
                    for (int i = 0; i < n; ++i) {
                        ra += cas[(int64_t)i * k & (n - 1)] * a[i];
                        rb += cas[(int64_t)i * k & (n - 1)] * b[i];
                    }
                    const double da = 0.5 * ((z[k].real() + z[m].real()) - (z[k].imag() - z[m].imag()));
                    const double db = 0.5 * ((z[k].imag() + z[m].imag()) + (z[k].real() - z[m].real()));
                    const long double fa = fx_to((fx_t)hx, q) - ra, fb = fx_to((fx_t)hy, q) - rb;
                    ef += fa * fa + fb * fb;
                    ed += (da - ra) * (da - ra) + (db - rb) * (db - rb);
                    norm += ra * ra + rb * rb;
                }
            }
            std::printf("%d %d %.3e %.3e\n", p, kind, (double)sqrtl(ef / norm), (double)sqrtl(ed / norm));
        }
    }
    for (int i = 0; i < 200000; ++i) {   // conversions: exact for the row's largest binade
        const double x = N(g) * exp(10 * N(g));
        const unsigned E = (high(x) >> 20) & 0x7FFu;
        if (fx_to(fx_from(x, E), (int)E - FX_BITS) != x) { std::printf("conversion of %a\n", x); return 1; }
    }
    if (fx_from(0.0, 1000) != 0 || fx_from(-0.0, 1000) != 0 || fx_to(0, 1000) != 0.0) return 1;
}
