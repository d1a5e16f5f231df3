// One component of a unit direction, num / sqrt(s), as the curve tracing's
// direction computes it with sqrt and /.
#pragma once

// A warp's FP64 instruction takes 64 cycles, dependent or not, whatever the
// number of active lanes; the compiler's square root and division take about 9
// each, half of a stage.  Here 1/sqrt(s) comes from the FP32 pipe (about 5
// cycles an instruction): the hardware estimate r0 (within 2 ulp, 2^-22) and
// one second-order step on e = 1 - s r0^2.  Of s = sh + sl, sh holds the upper
// 24 bits and sl the other 29, rounded to 24 (2^-48 of s); e is of the size of
// 2^-21, so each rounding of its FMA residuals is at most 2^-45, and so is that
// of the step itself.  Together y is within 2^-43 of 1/sqrt(s) (2^-43.4 at worst
// in a search with r0 at 2 ulp).  Square root and quotient then follow
// Markstein's scheme (IBM J. Res. Dev. 34, 1990): an approximation, its
// residual by FMA, and one corrected rounding.  With y off by d the values
// rounded last are within 1.5 d^2 and d^2 of the true ones, 2^-85, so the result
// is the correctly rounded one, as sqrt and / give, unless a true value lies
// that close to a rounding boundary (one in 2^30); it is then the neighbour.
__device__ __forceinline__ double f32_widen(float x)  // exact for normal x, integer pipe
{
    const unsigned b = __float_as_uint(x);
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
}

// bad: set where sqrt(s) is not positive (0, negative or NaN)
__device__ __forceinline__ double unit_component(double num, double s, bool& bad)
{
    const unsigned hi = (unsigned)__double2hiint(s), lo = (unsigned)__double2loint(s);
    if (hi - (963u << 20) < (120u << 20)) {  // 2^-60 <= s < 2^60
        const float sh = __uint_as_float(__funnelshift_r(lo, hi, 29) - (384u << 23));
        const float sl = __uint2float_rn(lo & 0x1fffffffu) * __uint_as_float(((hi >> 20) - 1023u - 52u + 127u) << 23);
        const float r0 = rsqrtf(sh);
        const float p = r0 * r0, pe = __fmaf_rn(r0, r0, -p);
        const float t = sh * p, te = __fmaf_rn(sh, p, -t);
        float e = (1.0f - t) - te;
        e = __fmaf_rn(-sh, pe, e);
        e = __fmaf_rn(-sl, p, e);
        const float rl = r0 * (e * __fmaf_rn(0.375f, e, 0.5f));
        double y = f32_widen(r0);
        if (fabsf(rl) >= 1.1754944e-38f) y = y + f32_widen(rl);
        const double hy = __hiloint2double(__double2hiint(y) - (1 << 20), __double2loint(y));  // y / 2
        double g = s * y;
        g = __fma_rn(__fma_rn(-g, g, s), hy, g);
        const double q = num * y;
        return __fma_rn(__fma_rn(-q, g, num), y, q);
    }
    const double nrm = sqrt(s);
    if (!(nrm > 0.0)) bad = true;
    return num / nrm;
}
