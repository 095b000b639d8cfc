// Host build of the fixed-point closures (csrc/fx64.cuh) with the library's
// own soil constants (make_fx_soil), for the CPU test of soils with n near 1.
#include <cmath>
#include <cstring>

#include "fx64.cuh"

using namespace rf;

static FxTables T;

extern "C" void fx_init()
{
    for (int j = 0; j < FX_TAB; j++) {
        const long double F = 1.0L + (long double)j / (long double)FX_TAB;
        T.rc[j] = (uint32_t)ceill(2147483648.0L / F);
        T.lg[j] = (uint64_t)rintl(-log2l((long double)T.rc[j] / 2147483648.0L) * 9223372036854775808.0L);
        T.e2[j] = (uint64_t)rintl(exp2l((long double)j / (long double)FX_TAB) * 9223372036854775808.0L);
    }
}

extern "C" int fx_takes_soil(double alpha, double n) { return make_fx_soil(true, alpha, n, 1.0 - 1.0 / n).ok; }

extern "C" void fx_eval(double alpha, double n, const double *h, int N, double *se, double *k, double *c)
{
    const FxSoil s = make_fx_soil(true, alpha, n, 1.0 - 1.0 / n);
    for (int i = 0; i < N; i++) {
        const double a = -h[i];
        uint64_t hb, r[3];
        std::memcpy(&hb, &a, 8);
        if (!fx_closure_vg(s, hb, &T, r[0], r[1], r[2])) {
            se[i] = k[i] = c[i] = NAN;
            continue;
        }
        std::memcpy(&se[i], &r[0], 8);
        std::memcpy(&k[i], &r[1], 8);
        std::memcpy(&c[i], &r[2], 8);
    }
}
