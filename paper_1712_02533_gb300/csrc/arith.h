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
