// Host check of the rows at the bottom of the exponent range: zeros go to the
// fixed-point form and stay zeros, nonzero subnormals do not.
#include <cstdio>
#include <cstring>

#include "rve_fixed.cuh"
using namespace rve;

int main() {
    auto exponent = [](double x) {
        uint64_t u;
        std::memcpy(&u, &x, 8);
        return fx_row_exponent(fx_high((unsigned)(u >> 32), (unsigned)u));
    };
    bool ok = fx_takes(exponent(0.0)) && fx_takes(exponent(-0.0)) && fx_takes(exponent(1.0));
    for (double x : {0x1p-1074, -0x1p-1074, 0x1p-1043, 0x1.8p-1042, 0x1p-1023, 0x1p-1022, 0x1p-900})
        ok = ok && !fx_takes(exponent(x));
    for (double x : {0.0, -0.0}) ok = ok && fx_to(fx_from(x, exponent(x)), 1023 - FX_BITS) == 0.0;
    std::printf("%s\n", ok ? "ok" : "wrong");
    return !ok;
}
