// fx64.cuh -- the van Genuchten / Mualem closures in 64-bit fixed point.
//
// GB300's FP64 pipe issues 2 thread-operations per clock and SM, its integer
// pipes 64: one FP64 multiply-add takes the time of some thirty integer
// instructions, so 64-bit fixed point from 32 x 32 -> 64 multiplies is both
// faster than FP64 and more exact (up to 64 significant bits against 53).
// Everything between the head's bit pattern and the three packed results
// (Se, K/Ks, C/cfac) is integer arithmetic; k_closure's FP64 work falls from
// 106 instructions a cell to about five.
//
// With u = -alpha h and base-2 logarithms, y = n log2 u, x = u^n = 2^y:
//   A = log2(1 + x)   = max(y, 0) + s      s = log2(1 + 2^-|y|)
//   B = log2(1 + 1/x) = max(-y, 0) + s
//   Se = 2^(-m A),  (x/(1+x))^m = 2^(-m B) = ys,  1/(1+x) = 2^-A
//   K/Ks = Se^(1/2) (1 - ys)^2,   C/cfac = ys / (1+x) = 2^(-(m B + A))
// 1 - ys is formed with full relative precision: from the power series of
// 1 - 2^-q where q = m B < 2^-9 (dry soil), and s likewise from the series of
// log2(1 + x') where x' = 2^-|y| < 2^-9; both series are the tails of the
// table-driven functions below, with the table entry 1.  With a small m, q is
// small in wet soil too: below FX_M_SMALL it is carried as a significand and
// an exponent at every head (with q on the grid of 2^-57 K was off by 15 units
// of the last place at n = 1.01, by 160 at 1.001).
//
// Logarithm and power of two: table-driven argument reduction (P. T. P. Tang,
// ACM TOMS 15 (1989) 144-157 and 16 (1990) 378-400) with 512 entries and the
// Taylor series of log2(1 + r) and 2^g - 1, r, g in [0, 2^-9), each term
// carried to the bits that reach the result's 2^-62; table entries are taken
// at the left edge of their interval so that r and g are unsigned.
// "Qk" below: an unsigned 64-bit integer v stands for v 2^-k.
#pragma once

#include <math.h>
#include <stdint.h>

#ifdef __CUDACC__
#define RF_HD __host__ __device__ __forceinline__
#else
#define RF_HD inline
#endif

namespace rf {

constexpr int FX_BITS = 9;
constexpr int FX_TAB = 1 << FX_BITS;

struct FxTables {
    uint64_t lg[FX_TAB];   // -log2(rc_j 2^-31)                Q63
    uint64_t e2[FX_TAB];   // 2^(j/512)                        Q63
    uint32_t rc[FX_TAB];   // 1/(1 + j/512), rounded up        Q31
};

// Fixed-point copies of a soil's parameters (make_fx_soil); ok = 0 sends
// every cell of the soil to the general closure.
struct FxSoil {
    int64_t la;        // log2(alpha)  Q58
    uint64_t nm;       // n 2^-ne in [1, 2)  Q63
    uint64_t m;        // m  Q64 (exact: m >= 2^-12)
    uint64_t Lmax;     // largest |log2 u| with |y| < 60, Q58
    int ne;            // exponent of n
    int ea;            // floor(log2 alpha)
    int ok;
    int mz;            // leading zeros of m
};

constexpr int FX_M_SMALL = 4;   // m < 2^-FX_M_SMALL (n < 1.067): q as a significand and an exponent

// Host: the constants of a van Genuchten soil.  Others, and parameters for
// which a field would not fit its format, get ok = 0.
inline FxSoil make_fx_soil(bool vg, double alpha, double n, double m)
{
    FxSoil f{};
    const long double la = log2l((long double)alpha);
    f.ok = (vg && n < 16.0 && m >= 0x1p-12 && la > -20.0L && la < 20.0L) ? 1 : 0;
    if (!f.ok) return f;
    f.ne = ilogb(n);
    f.ea = ilogb(alpha);
    f.la = (int64_t)rintl(la * 288230376151711744.0L);                          // 2^58
    f.nm = (uint64_t)ldexpl((long double)n, 63 - f.ne);
    f.m = (uint64_t)rintl((long double)m * 18446744073709551616.0L);            // 2^64
    f.mz = -1 - ilogb(m);
    const long double Lm = 60.0L / (long double)n;
    f.Lmax = (uint64_t)((Lm < 31.5L ? Lm : 31.5L) * 288230376151711744.0L);
    return f;
}

// High 64 bits of a 64 x 64 product, at most 2 units low: the low x low
// product and one carry are left out (three 32 x 32 multiply-adds).
RF_HD uint64_t fx_mulhi(uint64_t a, uint64_t b)
{
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
    const uint64_t m1 = (uint64_t)al * bh, m2 = (uint64_t)ah * bl;
    return (uint64_t)ah * bh + (uint32_t)(m1 >> 32) + (uint32_t)(m2 >> 32);
}

RF_HD uint32_t fx_mulhi32(uint32_t a, uint32_t b)
{
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}

// High 64 bits of a 64 x 32 product times 2^32 (a b 2^-32).
RF_HD uint64_t fx_mul32(uint64_t a, uint32_t b)
{
    return (uint64_t)(uint32_t)(a >> 32) * b + (uint32_t)(((uint64_t)(uint32_t)a * b) >> 32);
}

RF_HD int fx_clz(uint64_t v)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return v ? __builtin_clzll(v) : 64;
#endif
}

// G(r) of log2(1 + r) = a r - r^2 G(r), a = log2 e, for r in [0, 2^-9) given
// as rs = r 2^71: G = a (1/2 - r/3 + r^2/4 - r^3/5 + r^4/6), Q64.
RF_HD uint64_t fx_log_g(uint64_t rs)
{
    const uint32_t t = (uint32_t)(rs >> 31);                                     // Q40
    const uint32_t j5 = 0x93bb6287u - (fx_mulhi32(t, 0x7b1c2771u) >> 8);         // a/5 - r a/6     Q33
    const uint32_t i4 = 0xb8aa3b29u - (fx_mulhi32(t, j5) >> 8);                  // a/4 - r (..)    Q33
    const uint64_t i3 = 0x7b1c2770e80ff5d2ULL - (fx_mul32(rs, i4) >> 8);         // a/3 - r (..)    Q64
    return 0xb8aa3b295c17f0bcULL - (fx_mulhi(rs, i3) >> 7);                      // a/2 - r (..)    Q64
}

constexpr uint64_t FX_LOG2E = 0xb8aa3b295c17f0bcULL;   // log2 e, Q63

// log2 of M (Q63, M in [1, 2)) as Q63.
RF_HD uint64_t fx_log2(uint64_t M, const FxTables *tab)
{
    const uint32_t j = (uint32_t)(M >> (63 - FX_BITS)) & (FX_TAB - 1);
    const uint32_t c = tab->rc[j];
    const uint64_t t0 = (uint64_t)(uint32_t)M * c;
    const uint64_t t1 = (uint64_t)(uint32_t)(M >> 32) * c + (uint32_t)(t0 >> 32);   // 1 + r  Q62
    const uint64_t rs = (t1 << 9) | ((uint32_t)t0 >> 23);                           // r 2^71 (the 1 shifts out)
    const uint64_t g = fx_log_g(rs);
    const uint64_t ar = fx_mulhi(rs, FX_LOG2E);                                     // Q70
    const uint64_t r2g = fx_mulhi(fx_mulhi(rs, rs), g);                             // Q78
    return tab->lg[j] + ((ar - (r2g >> 8) + 64) >> 7);
}

// ln2 (1 -+ ...): W of 2^g - 1 = g W(g) (NEG false) or 1 - 2^-g = g W(g) (NEG
// true), g in [0, 2^-9) given as gs = g 2^73: ln2 +- g (ln2^2/2 +- g (ln2^3/6
// +- g (ln2^4/24 +- g ln2^5/120))), Q64.
template <bool NEG>
RF_HD uint64_t fx_exp_w(uint64_t gs)
{
    const uint32_t t = (uint32_t)(gs >> 32);                                        // Q41
    const uint32_t d5 = fx_mulhi32(t, 0xaec40u);                                    // Q38
    const uint32_t j4 = NEG ? 0x9d955b7eu - d5 : 0x9d955b7eu + d5;                  // Q38
    const uint32_t d4 = fx_mulhi32(t, j4) >> 11;
    const uint32_t i3 = NEG ? 0xe35846b9u - d4 : 0xe35846b9u + d4;                  // Q36
    const uint64_t d3 = fx_mul32(gs, i3) >> 13;
    const uint64_t h = NEG ? 0x3d7f7bff058b1d51ULL - d3 : 0x3d7f7bff058b1d51ULL + d3;   // Q64
    const uint64_t d2 = fx_mulhi(gs, h) >> 9;
    return NEG ? 0xb17217f7d1cf79acULL - d2 : 0xb17217f7d1cf79acULL + d2;
}

// 2^F for F in [0, 1) (Q64) as Q63 in [1, 2).
RF_HD uint64_t fx_exp2(uint64_t F, const FxTables *tab)
{
    const uint32_t j = (uint32_t)(F >> (64 - FX_BITS));
    const uint64_t gs = F << FX_BITS;                                               // g 2^73
    const uint64_t p = fx_mulhi(gs, fx_exp_w<false>(gs));                           // 2^g - 1  Q73
    const uint64_t T = tab->e2[j];
    return T + ((fx_mulhi(T, p) + 256) >> 9);
}

// The double M 2^e for M in Q63 with its top bit set (rounded to nearest);
// e within the normal range.
RF_HD uint64_t fx_pack(uint64_t M, int e)
{
    return ((uint64_t)(uint32_t)(e + 1022) << 52) + (M >> 11) + ((M >> 10) & 1);
}

// 1 - 2^-q = om 2^(eo - 63) for q = m (Bm 2^(eb - 62)), m < 2^-FX_M_SMALL, Bm
// below 2^63 and the product below 4; mB: q as Q57.
RF_HD void fx_one_minus_ys_small_m(const FxSoil &s, uint64_t Bm, int eb, uint64_t mB, const FxTables *tab,
                                   uint64_t &om, int &eo)
{
    const int zb = fx_clz(Bm);
    const uint64_t qm = fx_mulhi(Bm << zb, s.m << s.mz);                            // [2^62, 2^64)
    const int eq = eb - zb - s.mz;                                                  // q = qm 2^(eq - 62)
    const uint64_t q63 = eq <= -1 ? qm >> (eq < -64 ? 63 : -1 - eq) : ~0ULL;        // q  Q63 where q < 2
    if (q63 < 1ULL << 54) {                                                         // q < 2^-9
        const int sh = eq + 11;
        const uint64_t gs = sh >= 0 ? qm << sh : qm >> (sh < -63 ? 63 : -sh);       // q 2^73
        om = fx_mulhi(qm, fx_exp_w<true>(gs));
        eo = eq + 1;
        return;
    }
    eo = -1;
    if (q63 >> 63) {                                                                // q >= 1: the bits of Q57 do
        const int64_t z = -(int64_t)mB;
        om = 0 - (fx_exp2((uint64_t)z << 7, tab) >> (-(int)(z >> 57) - 1));
    } else {
        om = 0 - fx_exp2((0x8000000000000000ULL - q63) << 1, tab);                  // 2^-q = 2^(1 - q) / 2
    }
}

// Se, K/Ks and C/cfac (bit patterns of doubles) at |h| = the double with bits
// hb, h < 0.  Returns false, without results, when the state is outside the
// range of the fixed-point form (|log2 u| >= 31 or |y| >= 60; zero,
// subnormal and non-finite heads among them).
RF_HD bool fx_closure_vg(const FxSoil &s, uint64_t hb, const FxTables *tab, uint64_t &se_o, uint64_t &k_o,
                         uint64_t &c_o)
{
    const int E = (int)(hb >> 52) - 1023;
    if (!s.ok || (unsigned)(E + s.ea + 30) > 59u) return false;
    // L = log2 u, Q58
    const uint64_t lm = fx_log2((hb << 11) | 0x8000000000000000ULL, tab);
    const int64_t L = ((int64_t)E << 58) + (int64_t)(lm >> 5) + s.la;
    const bool dry = L >= 0;
    const uint64_t aL = dry ? (uint64_t)L : (uint64_t)(-L);
    if (aL > s.Lmax) return false;
    const uint64_t ay = (fx_mulhi(aL, s.nm) + 1) << s.ne;                                // |y|  Q57
    // x' = 2^-|y| = X 2^(e1 - 63)
    const int64_t z1 = -(int64_t)ay;
    const int e1 = (int)(z1 >> 57);                                                 // <= 0
    const uint64_t X = fx_exp2((uint64_t)z1 << 7, tab);
    // s = log2(1 + x') as s63 (Q63) and, with relative precision, sm 2^(es - 62)
    uint64_t s63, sm;
    int es;
    if (e1 >= -9) {
        const uint64_t v = e1 == 0 ? 0x7fffffffffffffffULL : X >> (-e1);
        s63 = fx_log2(0x8000000000000000ULL + v, tab);
        sm = s63;
        es = -1;
    } else {
        const uint64_t rs = X >> (-e1 - 8);                                         // x' 2^71
        const uint64_t q = FX_LOG2E - (fx_mulhi(rs, fx_log_g(rs)) >> 8);            // s / x'  Q63
        sm = fx_mulhi(X, q);
        es = e1;
        s63 = sm >> (-e1 - 1);
    }
    const uint64_t s57 = s63 >> 6;
    const uint64_t A = dry ? ay + s57 : s57, B = dry ? s57 : ay + s57;              // Q57
    const uint64_t mA = fx_mulhi(A, s.m) + 1, mB = fx_mulhi(B, s.m) + 1;           // + 1: mean of fx_mulhi
    // Se^(1/2) = 2^(-mA/2): mA is Q57, so -mA/2 is the same integer in Q58
    const int64_t z2 = -(int64_t)mA;
    const int eq = (int)(z2 >> 58);
    const uint64_t Q = fx_exp2((uint64_t)z2 << 6, tab);
    const uint64_t Q2 = fx_mulhi(Q, Q);                                             // Q62, [1, 4)
    se_o = (Q2 >> 63) ? fx_pack(Q2, 2 * eq + 1) : fx_pack(Q2 << 1, 2 * eq);
    // C/cfac = 2^-(mB + A)
    const int64_t z3 = -(int64_t)(mB + A);
    c_o = fx_pack(fx_exp2((uint64_t)z3 << 7, tab), (int)(z3 >> 57));
    // 1 - ys = om 2^(eo - 63)
    const uint64_t q63 = fx_mulhi(s63, s.m);                                        // m s  Q63
    uint64_t om;
    int eo;
    if (s.mz >= FX_M_SMALL) {
        fx_one_minus_ys_small_m(s, dry ? sm : B, dry ? es : 5, mB, tab, om, eo);    // B 2^-57 = B 2^(5 - 62)
    } else if (dry && q63 < (1ULL << 54) - 8) {   // margin: fx_mulhi may be 2 units low
        const int zs = fx_clz(sm);
        const uint64_t qm = fx_mulhi(sm << zs, s.m);                                // q = qm 2^(es - 62) < 2^-9
        es -= zs;
        const int sh = es + 11;
        const uint64_t gs = sh >= 0 ? qm << sh : qm >> (sh < -63 ? 63 : -sh);       // q 2^73
        om = fx_mulhi(qm, fx_exp_w<true>(gs));
        eo = es + 1;
    } else {
        // 2^-q, q = mB; dry: q = m s < 1 with the bits of Q63
        const int64_t z4 = -(int64_t)mB;
        const int e4 = dry ? -1 : (int)(z4 >> 57);
        const uint64_t F = dry ? (0x8000000000000000ULL - q63) << 1 : (uint64_t)z4 << 7;
        om = 0 - (fx_exp2(F, tab) >> (-e4 - 1 > 63 ? 63 : -e4 - 1));                // Q64
        eo = -1;
    }
    const int zo = fx_clz(om);
    om <<= zo;
    eo -= zo;
    const uint64_t kk = fx_mulhi(fx_mulhi(om, om), Q);                              // Q61, [1/..: 2^61, 2^64)
    const int zk = fx_clz(kk);
    k_o = fx_pack(kk << zk, eq + 2 * eo + 2 - zk);
    return true;
}

}  // namespace rf
