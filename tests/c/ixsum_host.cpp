// Host build of the integer sums (csrc/ix_sum.cuh) for the CPU test: the
// same limbs, warp by warp, with the warp reductions as loops.
#include <cstring>

#include "ix64.cuh"
#include "ix_sum.cuh"

using namespace rf;

static IxSum warp_sum(const double *v, int n)
{
    IxSum s{0, {0, 0, 0}};
    uint64_t b[32] = {};
    for (int i = 0; i < n; i++) {
        std::memcpy(&b[i], &v[i], 8);
        if (ix_exp(b[i]) > s.e) s.e = ix_exp(b[i]);
    }
    if (s.e == 0x7ff) {
        for (int i = 0; i < 32; i++)
            if (ix_exp(b[i]) == 0x7ff) s.l[0] |= (int32_t)ix_special(b[i]);
        return s;
    }
    s.e = s.e ? s.e : 1;
    for (int i = 0; i < 32; i++) {
        int32_t l[3];
        ix_limbs(b[i], s.e, l);
        for (int k = 0; k < 3; k++)
            if (__builtin_add_overflow(s.l[k], l[k], &s.l[k])) __builtin_trap();
    }
    return s;
}

// Sum of one warp's n <= 32 values.
extern "C" double ix_sum32(const double *v, int n)
{
    const IxSum s = warp_sum(v, n);
    const uint64_t r = s.e == 0x7ff ? ix_special_bits((uint32_t)s.l[0]) : ix_round(s.e, ix_join(s));
    double d;
    std::memcpy(&d, &r, 8);
    return d;
}

// Sum of seven values >= 0; NaN when the integer form refuses them.
extern "C" double ix_sum_seven(const double *v)
{
    uint64_t b[7], s = 0x7ff8000000000000ULL;
    std::memcpy(b, v, sizeof b);
    ix_sum7(b, s);
    double d;
    std::memcpy(&d, &s, 8);
    return d;
}
