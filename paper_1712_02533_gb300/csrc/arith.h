// Float-pair arithmetic of the kernels, for host and device alike (the tests measure
// its errors on the host; compile with -ffp-contract=off there).
#pragma once
#include <math.h>

#include "tile_rows.h"

// Explicitly rounded on the device: the compiler must not contract them into FMAs.
REG_HD float add_rn(float a, float b)
{
#ifdef __CUDA_ARCH__
    return __fadd_rn(a, b);
#else
    return a + b;
#endif
}
REG_HD float sub_rn(float a, float b)
{
#ifdef __CUDA_ARCH__
    return __fsub_rn(a, b);
#else
    return a - b;
#endif
}
REG_HD float mul_rn(float a, float b)
{
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    return a * b;
#endif
}
REG_HD double add_rn(double a, double b)
{
#ifdef __CUDA_ARCH__
    return __dadd_rn(a, b);
#else
    return a + b;
#endif
}
REG_HD double mul_rn(double a, double b)
{
#ifdef __CUDA_ARCH__
    return __dmul_rn(a, b);
#else
    return a * b;
#endif
}

// a + b = s + e exactly.
REG_HD void two_sum(float a, float b, float &s, float &e)
{
    s = add_rn(a, b);
    float bb = sub_rn(s, a);
    e = add_rn(sub_rn(a, sub_rn(s, bb)), sub_rn(b, bb));
}

// A sum of products v_k s_k (s_k a double as two floats) as an unevaluated pair hi + lo.
// After every second product the pair is folded, so that lo stays below 3 ulp of hi and
// a product's rounding below 2^-46 of the largest partial sum: with M = sum |v_k s_k|
// the m products' sum is within (m 2^-45.5 + 2^-44) M.  (Never folded, lo grows with m
// and its rounding with m^2.)
struct PairSum {
    float hi = 0.f, lo = 0.f, mag = 0.f;
    REG_HD void add(float v, float sh, float sl)
    {
        const float p = mul_rn(v, sh), pl = fmaf(v, sl, fmaf(v, sh, -p));
        float e;
        two_sum(hi, p, hi, e);
        lo = add_rn(lo, add_rn(e, pl));
        mag = add_rn(mag, fabsf(p));
    }
    REG_HD void fold()
    {
        const float s = add_rn(hi, lo);
        lo = sub_rn(lo, sub_rn(s, hi));
        hi = s;
    }
    // What the sum plus a constant, times a factor (both doubles as two floats, the
    // factor positive), may be off after m products: the bound above and the roundings
    // of this end, doubled for those of mag and of the sums in double it stands for.
    REG_HD float tolerance(int m, float ch, float fh) const
    {
        return mul_rn(mul_rn(add_rn(mag, fabsf(ch)), fh), (float)(m + 4) * 2.8421709430404007e-14f);  // 2^-45
    }
    // (sum + constant) factor as two floats.
    REG_HD void scaled(float ch, float cl, float fh, float fl, float &ph, float &pl) const
    {
        float t, te;
        two_sum(hi, ch, t, te);
        te = add_rn(te, add_rn(lo, cl));
        ph = mul_rn(t, fh);
        pl = fmaf(t, fl, fmaf(te, fh, fmaf(t, fh, -ph)));
    }
};

// 1 / sqrt(v) as an unevaluated pair r + lo from a float value r0 of it (rsqrtf: within
// 2 ulp), v within float's range: one third-order step (Halley's iteration for v^-1/2),
// whose residual 1 - v r0^2 carries the rounding of v r0.  r is the pair rounded; what
// the step leaves is below 2^-63.
struct RootInv {
    double r, lo;
};
REG_HD RootInv rsqrt_step(double v, float r0)
{
    const double r = (double)r0, t = mul_rn(v, r), tl = fma(v, r, -t);
    const double e = fma(-tl, r, fma(-t, r, 1.0)), re = r * e, c = fma(e, 0.375, 0.5);
    RootInv q;
    q.r = fma(re, c, r);
    q.lo = fma(re, c, r - q.r);
    return q;
}

// s / sqrt(v), and sqrt(v) for s = v, rounded once (a square root and a division round
// twice: up to 2 2^-53 off).
REG_HD double times(double s, const RootInv &q)
{
    const double p = mul_rn(s, q.r);
    return add_rn(p, fma(s, q.lo, fma(s, q.r, -p)));
}
