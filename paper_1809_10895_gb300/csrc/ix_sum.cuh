// ix_sum.cuh -- sums of doubles over warps and blocks on the integer pipes.
//
// An FP64 warp instruction holds a quarter of an SM for 64 cycles, so the tail
// of a block sum (eight values a lane, then five exchanges) takes 1150 cycles.
// Here a value becomes three signed 26-bit limbs of its significand, shifted to
// the warp's largest exponent, and three integer warp reductions add them: the
// sum of a warp is exact but for bits below 2^-77 of its largest term, that of
// a block is rounded to a double once.
//
// Sum of doubles: U 2^(e - 1100), e the largest exponent field (at least 1).
#pragma once

#include "fx64.cuh"

namespace rf {

struct IxSum {
    uint32_t e;              // exponent field; 0x7ff: l[0] = 1 (NaN) | 2 (+inf) | 4 (-inf)
    int32_t l[3];            // 26-bit limbs from the lowest
};

RF_HD uint32_t ix_exp(uint64_t b) { return (uint32_t)(b >> 52) & 0x7ffu; }

// Limbs of the double with bits b (finite) at exponent e >= its own.
RF_HD void ix_limbs(uint64_t b, uint32_t e, int32_t (&l)[3])
{
    const uint32_t ex = ix_exp(b);
    const uint64_t m = (b & 0xfffffffffffffULL) | (ex ? 1ULL << 52 : 0);
    const uint32_t sh = e - (ex ? ex : 1u);
    const uint32_t s2 = sh + 27 < 63 ? sh + 27 : 63, s1 = sh + 1 < 63 ? sh + 1 : 63;
    const uint32_t s0 = sh < 25 ? 25 - sh : 0, r0 = sh < 25 ? 0 : sh - 25 < 63 ? sh - 25 : 63;
    const int32_t sg = (int32_t)(b >> 32) >> 31;              // 0 or -1
    l[2] = ((int32_t)(m >> s2) ^ sg) - sg;
    l[1] = ((int32_t)((m >> s1) & 0x3ffffff) ^ sg) - sg;
    l[0] = ((int32_t)(((m << s0) >> r0) & 0x3ffffff) ^ sg) - sg;
}

// What an infinite or NaN term means for the sum.
RF_HD uint32_t ix_special(uint64_t b)
{
    return (b & 0xfffffffffffffULL) ? 1u : (b >> 63) ? 4u : 2u;
}

RF_HD __int128 ix_join(const IxSum &s)
{
    return ((__int128)s.l[2] << 52) + (((int64_t)s.l[1] << 26) + s.l[0]);
}

// Bits of the double nearest to U 2^(e - 1100) (ties to even).
RF_HD uint64_t ix_round(uint32_t e, __int128 U)
{
    if (U == 0) return 0;
    const uint64_t sign = U < 0 ? 1ULL << 63 : 0;
    const unsigned __int128 a = U < 0 ? -(unsigned __int128)U : (unsigned __int128)U;
    uint64_t hi = (uint64_t)(a >> 64), lo = (uint64_t)a;
    int n = 0;                                                // leading zeros
    if (hi == 0) {
        hi = lo;
        lo = 0;
        n = 64;
    }
    const int z = fx_clz(hi);
    if (z) {
        hi = (hi << z) | (lo >> (64 - z));
        lo <<= z;
    }
    n += z;
    const int ef = (int)e + 50 - n;                           // exponent field
    if (ef >= 0x7ff) return sign | (0x7ffULL << 52);
    int drop = 11;
    if (ef < 1) drop = 12 - ef < 63 ? 12 - ef : 63;           // subnormal
    const uint64_t rem = (hi << (64 - drop)) | (lo != 0), half = 1ULL << 63;
    uint64_t r = hi >> drop;
    if (ef >= 1) r += (uint64_t)(ef - 1) << 52;
    r += rem > half || (rem == half && (r & 1));
    return sign | r;
}

// Bits of the infinity or NaN that special terms sum to.
RF_HD uint64_t ix_special_bits(uint32_t code)
{
    return (code & 1u) || code == 6u ? 0x7ff8000000000000ULL : code == 2u ? 0x7ff0000000000000ULL
                                                                          : 0xfff0000000000000ULL;
}

#ifdef __CUDACC__
// Maximum over the warp, on every lane.
__device__ __forceinline__ uint64_t ix_warp_max(uint64_t b)
{
    const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(b >> 32));
    const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(b >> 32) == hi ? (uint32_t)b : 0u);
    return (uint64_t)hi << 32 | lo;
}

// Sum of a double over the warp, on every lane.
__device__ __forceinline__ IxSum ix_warp_sum(double v)
{
    const uint64_t b = (uint64_t)__double_as_longlong(v);
    IxSum s;
    s.e = __reduce_max_sync(0xffffffffu, ix_exp(b));
    if (s.e == 0x7ffu) {
        s.l[0] = (int)__reduce_or_sync(0xffffffffu, ix_exp(b) == 0x7ffu ? ix_special(b) : 0u);
        s.l[1] = s.l[2] = 0;
        return s;
    }
    s.e = s.e ? s.e : 1u;
    int32_t l[3];
    ix_limbs(b, s.e, l);
#pragma unroll
    for (int i = 0; i < 3; i++) s.l[i] = __reduce_add_sync(0xffffffffu, l[i]);
    return s;
}

__device__ __forceinline__ double ix_double(const IxSum &s)
{
    return __longlong_as_double(
        (long long)(s.e == 0x7ffu ? ix_special_bits((uint32_t)s.l[0]) : ix_round(s.e, ix_join(s))));
}

// Sum over the warp of up to eight lanes' sums (the others pass e = 0, l = 0),
// rounded, on every lane.
__device__ __forceinline__ double ix_fold8(const IxSum &s)
{
    const uint32_t e = __reduce_max_sync(0xffffffffu, s.e);
    if (e == 0x7ffu)
        return __longlong_as_double((long long)ix_special_bits(
            __reduce_or_sync(0xffffffffu, s.e == 0x7ffu ? (uint32_t)s.l[0] : 0u)));
    const uint32_t d = e - s.e;
    const __int128 t = d < 127 ? ix_join(s) >> d : 0;         // |t| < 2^83
    const uint64_t lo = (uint64_t)t;
    const int32_t l0 = (int32_t)(lo & 0xfffffff), l1 = (int32_t)((lo >> 28) & 0xfffffff), l2 = (int32_t)(t >> 56);
    const __int128 U = ((__int128)__reduce_add_sync(0xffffffffu, l2) << 56) +
                       (((int64_t)__reduce_add_sync(0xffffffffu, l1) << 28) + __reduce_add_sync(0xffffffffu, l0));
    return __longlong_as_double((long long)ix_round(e, U));
}
#endif

}  // namespace rf
