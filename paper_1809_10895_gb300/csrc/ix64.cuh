// ix64.cuh -- FP64 operations on positive operands by integer arithmetic.
//
// GB300's FP64 pipe issues 2 thread-operations per clock and SM, so an add
// holds it as long as some thirty integer instructions take.  Sums, scalings
// and reciprocals of positive numbers need no cancellation handling and are
// cheap on mantissas and exponents; the assembly runs them beside the FP64
// pipe instead of on it.  Results are within 0.51 units of the last place.
// A number is (M, e): M 2^(e - 63) with M's top bit set, or M = 0.
#pragma once

#include <math.h>

#include "fx64.cuh"

namespace rf {

struct IxNum {
    uint64_t M;
    int e;
};

// A positive normal double's bits.
RF_HD IxNum ix_unpack(uint64_t b)
{
    return IxNum{(b << 11) | 0x8000000000000000ULL, (int)(b >> 52) - 1023};
}

// (a + b) c for normalised a, b, c > 0.
RF_HD IxNum ix_add_mul(IxNum a, IxNum b, IxNum c)
{
    const bool sw = a.e < b.e;
    const int eb = sw ? b.e : a.e;
    int d = eb - (sw ? a.e : b.e);
    const uint64_t mb = sw ? b.M : a.M, ms = sw ? a.M : b.M;
    d = d > 62 ? 62 : d;
    uint64_t p = fx_mulhi((mb >> 1) + (ms >> (d + 1)), c.M);      // [2^61, 2^64)
    int e = eb + c.e + 2;
    if (!(p >> 63)) { p <<= 1; e--; }
    if (!(p >> 63)) { p <<= 1; e--; }
    return IxNum{p, e};
}

RF_HD IxNum ix_add(IxNum a, IxNum b)
{
    const bool sw = a.e < b.e;
    int d = sw ? b.e - a.e : a.e - b.e;
    const uint64_t mb = sw ? b.M : a.M, ms = sw ? a.M : b.M;
    d = d > 62 ? 62 : d;
    uint64_t p = (mb >> 1) + (ms >> (d + 1));                      // [2^62, 2^64)
    int e = (sw ? b.e : a.e) + 1;
    if (!(p >> 63)) { p <<= 1; e--; }
    return IxNum{p, e};
}

RF_HD uint64_t ix_pack(IxNum a) { return fx_pack(a.M, a.e); }

// Sum of seven doubles >= 0 (bits b), zeros among them: significands shifted
// to the largest exponent with three bits of headroom, one rounding.  False,
// without a result, when a term is negative or not finite or none exceeds
// 2^-900.
RF_HD bool ix_sum7(const uint64_t (&b)[7], uint64_t &sum)
{
    uint32_t top = 0;
    for (int i = 0; i < 7; i++) top = top > (uint32_t)(b[i] >> 32) ? top : (uint32_t)(b[i] >> 32);
    top >>= 20;
    if (top - 123u > 1900u) return false;
    uint64_t s = 0;
    for (int i = 0; i < 7; i++) {
        uint32_t d = top + 3 - (uint32_t)(b[i] >> 52);     // zeros and subnormals: more than 63
        d = d < 63 ? d : 63;
        s += ((b[i] << 11) | 0x8000000000000000ULL) >> d;
    }
    const int z = fx_clz(s);                               // 0 to 3
    sum = fx_pack(s << z, (int)top - 1020 - z);
    return true;
}

// The float (bits) whose reciprocal is estimated for M in [1, 2) (Q63): M's
// leading bits with the last three set to 2, so that an estimate off by up to
// 2^-23 lies in [1/2, 1) however close M is to 1 or 2.
RF_HD uint32_t ix_rcp_arg(uint64_t M) { return ((uint32_t)(M >> 40) & 0x7ffff8u) | 0x3f800002u; }

// 1/M, Q64 in (0.5, 1), from the estimate (bits rb): ri (1 + e + e^2) with ri
// the estimate (Q32) and |e| = |1 - M ri| <= 2^-20 (6 + 2 units of 2^-23); e^3
// is below 0.008 units of a double's last place.
RF_HD uint64_t ix_rcp_refine(uint64_t M, uint32_t rb)
{
    const uint32_t ri = (rb << 8) | 0x80000000u;
    const int64_t e = (int64_t)(0x8000000000000000ULL - fx_mul32(M, ri));                             // Q63
    const int32_t es = (int32_t)(e >> 13);                                                            // Q50
    const int64_t s = e + (((int64_t)es * es) >> 37);                                                 // e + e^2
    const int64_t t = (int64_t)(int32_t)(s >> 32) * ri + (int64_t)(uint32_t)(((uint64_t)(uint32_t)s * ri) >> 32);
    return ((uint64_t)ri << 32) + (uint64_t)(t << 1);
}

// a r 2^(-eb), r = 1/M of a number M 2^eb (ix_rcp).
RF_HD uint64_t ix_quot(IxNum a, uint64_t r, int eb)
{
    uint64_t q = fx_mulhi(a.M, r);                                 // [2^62, 2^64)
    const int up = (int)(q >> 63);
    q = up ? q : q << 1;
    return fx_pack(q, a.e - eb - 1 + up);
}

// Exponents for which quotients stay normal (a negative number's sign bit
// fails the test).
RF_HD bool ix_quot_ok(uint64_t a, uint64_t b)
{
    return (uint32_t)(a >> 52) - 700u < 650u && (uint32_t)(b >> 52) - 700u < 650u;
}

// The bits of the float nearest to the double with bits b (ties to even);
// not where it is zero, subnormal, infinite or NaN as a float.
RF_HD bool ix_d2f_ok(uint64_t b) { return ((uint32_t)(b >> 52) & 0x7ffu) - 897u <= 253u; }
RF_HD uint32_t ix_d2f_bits(uint64_t b)
{
    const uint64_t v = (b & 0x7fffffffffffffffULL) - (896ULL << 52);
    return (uint32_t)((v + 0x0fffffffULL + ((v >> 29) & 1)) >> 29) | ((uint32_t)(b >> 32) & 0x80000000u);
}

// The bits of the float with bits b as a double; not where it is subnormal,
// infinite or NaN.
RF_HD bool ix_f2d_ok(uint32_t b)
{
    const uint32_t m = b & 0x7fffffffu;
    return m - 0x00800000u < 0x7f000000u || !m;
}
RF_HD uint64_t ix_f2d_bits(uint32_t b)
{
    const uint32_t m = b & 0x7fffffffu;
    return (m ? ((uint64_t)m << 29) + (896ULL << 52) : 0) | (uint64_t)(b & 0x80000000u) << 32;
}

// Square root of a in [2^-99, 2^99], relative error below 2^-44: the float
// root s plus (a - s^2) / (2 s), of which only the difference and the sum need
// FP64 (an FP64 root is some fifteen dependent instructions of 64 cycles).
RF_HD double ix_root_step(double a, double s, float sf)
{
    return s + (double)((float)fma(-s, s, a) * (0.5f / sf));
}

#ifdef __CUDACC__
// 1/M for M in [1, 2) (Q63), Q64 in (0.5, 1).
__device__ __forceinline__ uint64_t ix_rcp(uint64_t M)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(ix_rcp_arg(M))));
    return ix_rcp_refine(M, __float_as_uint(r));
}

// The float nearest to a double (ties to even).
__device__ __forceinline__ float ix_d2f(double a)
{
    const uint64_t b = (uint64_t)__double_as_longlong(a);
    if (!ix_d2f_ok(b)) return (float)a;
    return __uint_as_float(ix_d2f_bits(b));
}

// Tests on the bits: a compare of doubles goes to the FP64 pipe.
__device__ __forceinline__ bool is_finite(double a)
{
    return ((uint32_t)__double2hiint(a) & 0x7ff00000u) != 0x7ff00000u;
}
__device__ __forceinline__ bool is_positive(double a)            // and no NaN
{
    return (unsigned long long)__double_as_longlong(a) - 1ULL < 0x7ff0000000000000ULL;
}
__device__ __forceinline__ bool not_above(double a, double b)    // a <= b, both >= 0 and no NaN
{
    return __double_as_longlong(a) <= __double_as_longlong(b);
}

// A float as a double.
__device__ __forceinline__ double ix_f2d(float a)
{
    const uint32_t b = __float_as_uint(a);
    if (!ix_f2d_ok(b)) return (double)a;
    return __longlong_as_double((long long)ix_f2d_bits(b));
}

// 1/a.
__device__ __forceinline__ double ix_rcp64(double a)
{
    const uint64_t b = (uint64_t)__double_as_longlong(a);
    if ((unsigned)(b >> 52) - 400u < 1200u) {
        const IxNum d = ix_unpack(b);
        return __longlong_as_double((long long)fx_pack(ix_rcp(d.M), -1 - d.e));
    }
    return 1.0 / a;
}

// Square root, relative error below 2^-44.
__device__ __forceinline__ double ix_sqrt(double a)
{
    if ((uint32_t)((uint64_t)__double_as_longlong(a) >> 52) - 924u >= 198u) return sqrt(a);
    const float sf = sqrtf(ix_d2f(a));
    return ix_root_step(a, ix_f2d(sf), sf);
}

// a/b.
__device__ __forceinline__ double ix_div(double a, double b)
{
    const uint64_t ab = (uint64_t)__double_as_longlong(a), bb = (uint64_t)__double_as_longlong(b);
    if (!ix_quot_ok(ab, bb)) return a / b;
    const IxNum d = ix_unpack(bb);
    return __longlong_as_double((long long)ix_quot(ix_unpack(ab), ix_rcp(d.M), d.e));
}
#endif

}  // namespace rf
