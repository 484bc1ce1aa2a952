// Host check of the rows that the fixed-point transforms take (csrc/rve_fixed.cuh)
// at both ends of the exponent range: the DC term of a constant row, the largest
// result there is, has to be the exact sum.  Prints every miss.
#include <cmath>
#include <cstdio>
#include <cstring>

#include "rve_fixed.cuh"
using namespace rve;

static unsigned high(double x) { uint64_t u; std::memcpy(&u, &x, 8); return (unsigned)(u >> 32); }

int main() {
    int misses = 0, taken = 0;
    for (int p = 5; p <= 11; ++p) {
        const int n = 1 << p;
        for (int e = -1022; e <= 1023; ++e) {
            for (double v : {std::ldexp(1.0, e), std::ldexp(-1.5, e), std::ldexp(std::nextafter(2.0, 0.0), e)}) {
                unsigned E = (high(v) >> 20) & 0x7FFu;
                if (!fx_takes(E)) continue;
                ++taken;
                const FxShifts f = fx_schedule(p, 2u * n * fx_size(high(v), E));
                E -= f.finer;
                // H_a(0) is n times the element, and comes doubled
                const __int128 dc = ((__int128)fx_from(v, E) * n) >> (fx_scale(p, f) - 1);
                const double h = fx_to((fx_t)dc, (int)E - FX_BITS + fx_scale(p, f) - 1);
                const double want = v * n;
                if (!(std::fabs(h - want) <= std::fabs(want) * 0x1p-52)) {
                    if (++misses < 10) std::printf("n %d: %d times %a gave %a\n", n, n, v, h);
                }
            }
        }
    }
    std::printf("%d rows taken, %d misses\n", taken, misses);
    return misses != 0 || taken < 7 * 3 * 1800;
}
