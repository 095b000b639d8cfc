// Host build of the integer forms of FP64 arithmetic (csrc/ix64.cuh) for the
// CPU test: the same source that the kernels include; the estimate of a
// reciprocal, an instruction there, is a rounded quotient `ulps` units off.
#include <cmath>
#include <cstring>

#include "ix64.cuh"

using namespace rf;

static uint64_t bits(double a)
{
    uint64_t b;
    std::memcpy(&b, &a, 8);
    return b;
}
static double value(uint64_t b)
{
    double a;
    std::memcpy(&a, &b, 8);
    return a;
}

static uint64_t rcp(uint64_t M, int ulps)
{
    const uint32_t xb = ix_rcp_arg(M);
    uint32_t rb;
    float x;
    std::memcpy(&x, &xb, 4);
    const float r = 1.0f / x + (float)ulps * 0x1p-24f;      // units of a result in [1/2, 1)
    std::memcpy(&rb, &r, 4);
    return ix_rcp_refine(M, rb);
}

extern "C" double ix_h_rcp(double a, int ulps)
{
    const IxNum d = ix_unpack(bits(a));
    return value(fx_pack(rcp(d.M, ulps), -1 - d.e));
}

// NaN where the integer form leaves the division to the instruction.
extern "C" double ix_h_div(double a, double b, int ulps)
{
    if (!ix_quot_ok(bits(a), bits(b))) return NAN;
    const IxNum d = ix_unpack(bits(b));
    return value(ix_quot(ix_unpack(bits(a)), rcp(d.M, ulps), d.e));
}

extern "C" double ix_h_add_mul(double a, double b, double c)
{
    return value(ix_pack(ix_add_mul(ix_unpack(bits(a)), ix_unpack(bits(b)), ix_unpack(bits(c)))));
}

extern "C" double ix_h_add(double a, double b) { return value(ix_pack(ix_add(ix_unpack(bits(a)), ix_unpack(bits(b))))); }

extern "C" double ix_h_sqrt(double a)
{
    const float s = sqrtf((float)a);
    return ix_root_step(a, (double)s, s);
}

// The FP32 reciprocal as the ensemble's Jacobi scaling forms it.
extern "C" float ix_h_rcp32(double a, int ulps)
{
    const double r = ix_h_rcp(a, ulps);
    const uint32_t f = ix_d2f_bits(bits(r));
    float v = NAN;
    if (ix_d2f_ok(bits(r))) std::memcpy(&v, &f, 4);
    return v;
}

// NaN where the integer form leaves the conversion to the instruction.
extern "C" float ix_h_d2f(double a)
{
    const uint32_t f = ix_d2f_bits(bits(a));
    float v = NAN;
    if (ix_d2f_ok(bits(a))) std::memcpy(&v, &f, 4);
    return v;
}

extern "C" double ix_h_f2d(float a)
{
    uint32_t b;
    std::memcpy(&b, &a, 4);
    return ix_f2d_ok(b) ? value(ix_f2d_bits(b)) : NAN;
}
