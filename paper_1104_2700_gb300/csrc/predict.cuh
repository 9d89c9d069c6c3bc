// The double-single predictor (Eqs. xpred, vpred) and the order-preserving
// time keys, shared by the predictor kernels and by the force kernel that
// predicts its own tiles.
#pragma once

#include <cstdint>

#include "nb_device.cuh"
#include "nb_launch.h"

namespace nb {

// Order-preserving map of doubles to unsigned 64-bit keys (for atomicMin).
__device__ __forceinline__ unsigned long long dkey(double x)
{
    const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double dkey_decode(unsigned long long k)
{
    const unsigned long long b = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    return __longlong_as_double(static_cast<long long>(b));
}

// ---------------------------------------------------------------------------
// Steps 2-3 for the precisions whose j layout holds double-single values
// (MIXED, DS, HYBRID): the prediction in double-single arithmetic on the
// FP32 pipes.  GB300 spends ~68 cycles on each FP64 warp instruction, and the
// FP64 Horner form plus the FP64 split into the layout took ~80 of them per
// particle, so over a large system (an ensemble predicts every particle at
// each block step) the predictor was FP64-bound.  Here each FP64 state value
// is cut into hi + lo floats with integer operations on its bits (hi: the
// leading 24 significand bits; lo: the remaining 29 rounded to a float, so
// hi + lo keeps ~48 bits), Eqs. xpred and vpred run as double-single Horner
// steps (FMA-based TwoProd and TwoSum), and the grid-aligned split is taken
// from the double-single result.  The layout agrees with an FP64 prediction
// to its own resolution (~2^-47 of the bound); values far outside the
// layout's range (|x| < 2^-60 or > 2^60, or not finite) take FP64
// conversions instead.
// ---------------------------------------------------------------------------
struct Dsf {
    float hi, lo;
};

__device__ __forceinline__ Dsf dsf_of(double x)
{
    // work on the two 32-bit words (tests on the whole 64-bit pattern would
    // become FP64 compares, which cost as much as the conversion they avoid)
    const unsigned hw = static_cast<unsigned>(__double2hiint(x));
    const unsigned lw = static_cast<unsigned>(__double2loint(x));
    const unsigned e = (hw >> 20) & 0x7ffu;
    if (e - (1023u - 60u) > 120u) {  // zero, |x| < 2^-60 or > 2^60, not finite
        if (((hw & 0x7fffffffu) | lw) == 0u) return {0.f, 0.f};
        const float hi = __double2float_rn(x);
        return {hi, __double2float_rn(x - static_cast<double>(hi))};
    }
    const unsigned sign = hw & 0x80000000u;
    // 52 significand bits: 20 in hw, 32 in lw; hi keeps the leading 23
    const float hi =
        __uint_as_float(sign | ((e - 1023u + 127u) << 23) | ((hw & 0xfffffu) << 3) | (lw >> 29));
    // the remaining 29 significand bits are worth rest * 2^(e - 1075)
    const unsigned rest = lw & 0x1fffffffu;
    const float lo = __uint2float_rn(rest) * __uint_as_float((e - 1075u + 127u) << 23);
    return {hi, sign ? -lo : lo};
}

__device__ __forceinline__ Dsf dsf_add(Dsf a, Dsf b)
{
    float s, e;
    two_sum(a.hi, b.hi, s, e);
    e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
    const float h = __fadd_rn(s, e);
    return {h, __fsub_rn(e, __fsub_rn(h, s))};
}

__device__ __forceinline__ Dsf dsf_fma(Dsf a, Dsf b, Dsf c)  // a b + c
{
    float p, e;
    two_prod(a.hi, b.hi, p, e);
    e = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, e));
    const float h = __fadd_rn(p, e);
    return dsf_add({h, __fsub_rn(e, __fsub_rn(h, p))}, c);
}

__device__ __forceinline__ Dsf dsf_scale(Dsf a, float pow2) { return {a.hi * pow2, a.lo * pow2}; }

// The grid quantum of grid_quantum() as floats, from the bound's bits.
__device__ __forceinline__ void grid_quantum_f(uint32_t bound_bits, float& q, float& inv_q)
{
    const int eb = static_cast<int>((bound_bits >> 23) & 0xff);
    int e;
    if (eb == 0 || eb == 255)
        frexp(2.0 * static_cast<double>(__uint_as_float(bound_bits)), &e);
    else
        e = eb - 125;  // 2B = (1.f / 2) 2^(eb - 125), 1.f / 2 in [0.5, 1)
    if (e < -100) e = -100;  // (both powers stay normal floats; such values travel in lo)
    q = ldexpf(1.f, e - 23);
    inv_q = ldexpf(1.f, 23 - e);
}

// x rounded to a multiple of q (hi) and the rest (lo); x.hi - hi is exact.  The
// rounding looks at x.hi alone, which lies within an ulp of x (at most q/2 while
// |x| is within twice the bound), so |lo| < q, not q/2 as in grid_split.
__device__ __forceinline__ void grid_split_ds(Dsf x, float q, float inv_q, float& hi, float& lo)
{
    hi = rintf(x.hi * inv_q) * q;
    lo = __fadd_rn(__fsub_rn(x.hi, hi), x.lo);
}

// One component of a particle predicted over h, in the form of the j layout:
// its position split on the layout's grid (quantum q, inverse iq) and its
// velocity in double-single.  Eqs. xpred, vpred:
// x + h (v + h (a / 2 + h j / 6)), v + h (a + h j / 2).
struct PredictedComp {
    float hi, lo;
    Dsf v;
};

__device__ __forceinline__ PredictedComp predict_component(double x0, double v0, double a0,
                                                           double j0, Dsf h, float q, float iq)
{
    PredictedComp p;
    const Dsf sixth = {0x1.555556p-3f, -0x1.555556p-28f};  // 1/6 to ~2^-50
    const Dsf x = dsf_of(x0), v = dsf_of(v0), a = dsf_of(a0), j = dsf_of(j0);
    Dsf u = dsf_fma(j, sixth, Dsf{0.f, 0.f});
    u = dsf_fma(h, u, dsf_scale(a, 0.5f));
    u = dsf_fma(h, u, v);
    grid_split_ds(dsf_fma(h, u, x), q, iq, p.hi, p.lo);
    p.v = dsf_fma(h, dsf_fma(h, dsf_scale(j, 0.5f), a), v);
    return p;
}

__device__ __forceinline__ Dsf dsf_mass(double G, double m)
{
    return dsf_fma(dsf_of(G), dsf_of(m), Dsf{0.f, 0.f});
}

// The layout's velocity split.  HYB: the FP32 value of v and the rest (far
// pairs difference FP32 velocities, near pairs the whole double-single value);
// DS: on the velocities' grid.
template <bool HYB>
__device__ __forceinline__ void split_velocity(Dsf v, float q, float iq, float& vh, float& vl)
{
    if (HYB) {
        vh = __fadd_rn(v.hi, v.lo);
        vl = __fadd_rn(__fsub_rn(v.hi, vh), v.lo);
    } else {
        grid_split_ds(v, q, iq, vh, vl);
    }
}

}  // namespace nb
