// Host build of the fixed-point closures (csrc/fx64.cuh) for the CPU test:
// the same source that the kernels include, with tables and soil constants
// filled as the library fills them.
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

extern "C" int fx_eval(double alpha, double n, const double *h, int N, double *se, double *k, double *c)
{
    const double m = 1.0 - 1.0 / n;
    const long double la = log2l((long double)alpha), Lm = 60.0L / (long double)n;
    FxSoil s{};
    s.ok = 1;
    s.ne = ilogb(n);
    s.ea = ilogb(alpha);
    s.la = (int64_t)rintl(la * 288230376151711744.0L);
    s.nm = (uint64_t)ldexpl((long double)n, 63 - s.ne);
    s.m = (uint64_t)rintl((long double)m * 18446744073709551616.0L);
    s.Lmax = (uint64_t)((Lm < 31.5L ? Lm : 31.5L) * 288230376151711744.0L);
    int out = 0;
    for (int i = 0; i < N; i++) {
        const double a = -h[i];
        uint64_t hb, r[3];
        std::memcpy(&hb, &a, 8);
        if (!fx_closure_vg(s, hb, &T, r[0], r[1], r[2])) {
            se[i] = k[i] = c[i] = NAN;
            out++;
            continue;
        }
        std::memcpy(&se[i], &r[0], 8);
        std::memcpy(&k[i], &r[1], 8);
        std::memcpy(&c[i], &r[2], 8);
    }
    return out;
}
