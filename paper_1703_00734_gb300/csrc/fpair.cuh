// fpair.cuh -- arithmetic on float pairs: a value is the unevaluated sum h + l of two floats with
// |l| <= ulp(h) / 2 (below ulp(h) from split(), which truncates), about 48 significant bits (Dekker
// 1971, Knuth's two-sum; with FMA the error of a product is one instruction).
//
// Why: on this GPU the FP64 pipe takes a warp instruction every 17 clocks per SM and the FP32
// pipes four every clock.  A multiply-add of pairs is 12 FP32 instructions (3.3 clocks), so the
// conditional draws of the reduced-precision modes, whose Gram sums carry 24 bits at most, run
// on the FP32 pipes at 48 bits.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "common.cuh"

namespace bmf {

struct __align__(8) fpair {
    float h, l;
};

// s + e = a + b exactly (Knuth).
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// h + l with |l| <= ulp(h) / 2 from h, l with |h| >= |l| (or h = 0).
__device__ __forceinline__ fpair renorm(float h, float l)
{
    const float s = __fadd_rn(h, l);
    return fpair{s, __fsub_rn(l, __fsub_rn(s, h))};
}
__device__ __forceinline__ fpair renorm(fpair a) { return renorm(a.h, a.l); }

__device__ __forceinline__ fpair pmul(fpair a, fpair b)
{
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, e);
    e = __fmaf_rn(a.l, b.h, e);
    return renorm(p, e);
}

// acc - a b for normalised a and b.  acc.l collects the error terms without being normalised
// (it stays far below acc's scale over a row's K terms): renorm the accumulator before it is used
// as a factor.
__device__ __forceinline__ fpair pfnma(fpair acc, fpair a, fpair b)
{
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, e);
    e = __fmaf_rn(a.l, b.h, e);
    const float s = __fsub_rn(acc.h, p);
    const float bb = __fsub_rn(s, acc.h);
    const float err = __fsub_rn(__fsub_rn(acc.h, __fsub_rn(s, bb)), __fadd_rn(p, bb));
    return fpair{s, __fadd_rn(acc.l, __fsub_rn(err, e))};
}

__device__ __forceinline__ fpair padd(fpair a, fpair b)
{
    float s, e;
    two_sum(a.h, b.h, s, e);
    return renorm(s, __fadd_rn(e, __fadd_rn(a.l, b.l)));
}

// prior + tau g, the entry of a conditional precision (or right-hand side): normalised.
__device__ __forceinline__ fpair passemble(fpair prior, fpair tau, fpair g)
{
    const float p = __fmul_rn(tau.h, g.h);
    float e = __fmaf_rn(tau.h, g.h, -p);
    e = __fmaf_rn(tau.h, g.l, e);
    e = __fmaf_rn(tau.l, g.h, e);
    float s, r;
    two_sum(prior.h, p, s, r);
    return renorm(s, __fadd_rn(r, __fadd_rn(prior.l, e)));
}

// 1 / sqrt(d) for a normalised pair d > 0 within 2^+-100: y0 from the FP32 unit, then
// y0 + y0 (r / 2 + 3 r^2 / 8) with r = 1 - d y0^2 taken to about 2^-45 (the cubic term is below
// 2^-60): relative error below 2^-44.
__device__ __forceinline__ fpair prsqrt(fpair d)
{
    const float y = rsqrtf(d.h);
    const float p = __fmul_rn(y, y);
    const float pe = __fmaf_rn(y, y, -p);
    const float q = __fmul_rn(d.h, p);
    float e = __fmaf_rn(d.h, p, -q);
    e = __fmaf_rn(d.h, pe, e);
    e = __fmaf_rn(d.l, p, e);
    const float r = __fsub_rn(__fsub_rn(1.0f, q), e);
    return renorm(y, __fmul_rn(y, __fmaf_rn(__fmul_rn(r, r), 0.375f, __fmul_rn(0.5f, r))));
}

// Ranges within which a pair keeps its 48 bits through the products and sums of a conditional
// draw, from the exponent field (infinities and NaN fall outside).  Any term below 2^70; a
// precision's diagonal from 2^-60; a right-hand side, a draw and the solutions of both triangular
// solves zero or from 2^-100 (a zero that is no underflow: between right-hand side and solution lie
// factors of at least 2^-35).  Rows outside take the FP64 path.
__device__ __forceinline__ bool pair_below(double x)
{
    return ((unsigned)__double2hiint(x) & 0x7fffffffu) < (1023u + 70u) << 20;
}
__device__ __forceinline__ bool pair_vector(double x)
{
    const unsigned u = (unsigned)__double2hiint(x) & 0x7fffffffu;
    return u - ((1023u - 100u) << 20) < 170u << 20 || (u | (unsigned)__double2loint(x)) == 0u;
}
__device__ __forceinline__ bool pair_vector(float h)
{
    const unsigned u = __float_as_uint(h) & 0x7fffffffu;
    return u - ((127u - 100u) << 23) < 170u << 23 || u == 0u;
}
__device__ __forceinline__ bool pair_diag(float h) { return h >= 0x1p-60f && h < 0x1p70f; }

// The top 24 bits of x and the following 24 as a pair, on the integer pipe (the conversion
// instructions between FP32 and FP64 run on the FP64 pipe): relative error below 2^-48 down to
// 2^-78; x below 2^-126 reads as zero.  Not normalised: h is truncated, so l has its sign and may be
// just below ulp(h); what takes it as a factor loses at most one of the 48 bits.  x must pass
// pair_below.
__device__ __forceinline__ fpair split(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned mag = hi & 0x7fffffffu, sign = hi & 0x80000000u;
    const unsigned keep = mag < (897u << 20) ? 0u : 0xffffffffu;
    // exponent rebased from 1023 to 127, then the top 23 fraction bits
    const unsigned f = __funnelshift_l(lo, mag - (896u << 20), 3) & keep;
    // the remaining 29 bits, an integer in units of 2^-52 of x's power of two
    const float m = __fmul_rn((float)(int)(lo & 0x1fffffffu), 0x1p-52f);
    return fpair{__uint_as_float(f | sign), __fmul_rn(m, __uint_as_float((f & 0x7f800000u) | sign))};
}

// The pair as a double: exact widenings on the integer pipe, one FP64 addition.
__device__ __forceinline__ double join(fpair a) { return widen(a.h) + widen(a.l); }

__device__ __forceinline__ fpair shfl_pair(fpair a, int src)
{
    return fpair{__shfl_sync(0xffffffffu, a.h, src), __shfl_sync(0xffffffffu, a.l, src)};
}

}  // namespace bmf
