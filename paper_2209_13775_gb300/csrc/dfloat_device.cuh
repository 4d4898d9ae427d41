// dfloat_device.cuh -- numbers as unevaluated sums of two FP32 values (about 48 bits), and the
// largest eigenvalue of a Cauchy-Green tensor in them.
//
// GB300 issues 128 FP32 operations per SM and cycle and 2 FP64 ones, so a chain of FP32 operations
// that stands in for an FP64 one is worth taking wherever the result does not have to carry 53 bits.
// The FTLE is such a result: it is an FP32 value, the logarithm of an eigenvalue whose relative error
// here, from the positions on, is at most 2^-44 (2^-44.5 over 6M gradients in random orientations), and
// 2^-44 / sqrt(d) where the two largest eigenvalues come together (d: df_eig_max3).  The caller takes FP64
// wherever that exceeds 2^-30 of the logarithm, a thirty-second of the half ulp by which the stored value is
// rounded.  lcs_ftle's lambda_max and C, which are FP64 outputs, do not come from here.
//
// The sums and products are the error-free transformations of Knuth (TwoSum), Dekker (Fast2Sum)
// and the FMA residual of a product, written with round-to-nearest intrinsics so that no product
// is contracted into a following sum.  The sums below bound the absolute error by 2^-46 of the
// larger operand, which is what the shifts and determinants here need.
#pragma once

struct dfl {
    float h, l;
};

__device__ __forceinline__ dfl df_two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}

// a + b for |a| >= |b| (or a = 0)
__device__ __forceinline__ dfl df_fast_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

__device__ __forceinline__ dfl df_two_prod(float a, float b)
{
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}

__device__ __forceinline__ dfl df_neg(dfl a) { return {-a.h, -a.l}; }

__device__ __forceinline__ dfl df_add(dfl a, dfl b)
{
    const dfl s = df_two_sum(a.h, b.h);
    return df_fast_sum(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}

__device__ __forceinline__ dfl df_sub(dfl a, dfl b) { return df_add(a, df_neg(b)); }

__device__ __forceinline__ dfl df_add(dfl a, float b)
{
    const dfl s = df_two_sum(a.h, b);
    return df_fast_sum(s.h, __fadd_rn(s.l, a.l));
}

__device__ __forceinline__ dfl df_mul(dfl a, dfl b)
{
    const dfl p = df_two_prod(a.h, b.h);
    return df_fast_sum(p.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, p.l)));
}

__device__ __forceinline__ dfl df_mul(dfl a, float b)
{
    const dfl p = df_two_prod(a.h, b);
    return df_fast_sum(p.h, __fmaf_rn(a.l, b, p.l));
}

// times a power of two (exact)
__device__ __forceinline__ dfl df_scale(dfl a, float s) { return {__fmul_rn(a.h, s), __fmul_rn(a.l, s)}; }

// sqrt(a), a >= 0
__device__ __forceinline__ dfl df_sqrt(dfl a)
{
    if (!(a.h > 0.0f)) return {a.h == 0.0f ? 0.0f : a.h - a.h, 0.0f};   // NaN stays NaN
    const float s = __fsqrt_rn(a.h);
    return df_fast_sum(s, __fdividef(__fadd_rn(__fmaf_rn(-s, s, a.h), a.l), s + s));
}

// the power of two 2^-e (and its inverse) that takes x = m 2^e into [1, 2); x normal
__device__ __forceinline__ float df_inv_pow2(float x, float &pow2)
{
    const unsigned e = __float_as_uint(x) & 0x7f800000u;
    pow2 = __uint_as_float(e);
    return __uint_as_float(0x7f000000u - e);
}

// 2x2 C = (a, b, c): lambda_max = (a + c)/2 + sqrt(((a - c)/2)^2 + b^2)
__device__ __forceinline__ dfl df_eig_max2(const dfl *C)
{
    float is;
    const float s = df_inv_pow2(fmaxf(C[0].h, C[2].h), is);
    const dfl a = df_scale(C[0], s), b = df_scale(C[1], s), c = df_scale(C[2], s);
    const dfl m = df_scale(df_add(a, c), 0.5f), d = df_scale(df_sub(a, c), 0.5f);
    return df_scale(df_add(m, df_sqrt(df_add(df_mul(d, d), df_mul(b, b)))), is);
}

// 3x3 packed C: lambda_max from the characteristic cubic of the shifted, normalised matrix
// (C - q I) / p, whose largest root solves beta^3 - 3 beta - 2 r = 0, r = det / 2 in [-1, 1].  With
// d = 1 - |r| and t the root in [0, 2 - sqrt 3] of 9 t - 6 t^2 + t^3 = 2 d (simple everywhere, its
// slope 3 (1 - t)(3 - t) is at least 5.9), beta = 2 - t for r >= 0; for r < 0 the isolated root is
// t - 2 and beta the larger root of the quadratic that is left, 1 - t/2 + sqrt(3 t (4 - t)) / 2.
// An error e of r moves that root by about e / sqrt(6 d): *gap is sqrt(d), 1 for r >= 0, and 0 below
// d = 1e-9, where d itself has lost its digits.  (0.25: all three eigenvalues within 2e-13 of q.)
__device__ __forceinline__ dfl df_eig_max3(const dfl *C, float *gap)
{
    float is;
    const float s = df_inv_pow2(fmaxf(C[0].h, fmaxf(C[3].h, C[5].h)), is);
    const dfl a00 = df_scale(C[0], s), a01 = df_scale(C[1], s), a02 = df_scale(C[2], s), a11 = df_scale(C[3], s),
              a12 = df_scale(C[4], s), a22 = df_scale(C[5], s);
    const dfl third = {0x1.555556p-2f, -0x1.555556p-27f};
    const dfl q = df_mul(df_add(df_add(a00, a11), a22), third);
    dfl b00 = df_sub(a00, q), b11 = df_sub(a11, q), b22 = df_sub(a22, q);
    const dfl off = df_add(df_add(df_mul(a01, a01), df_mul(a02, a02)), df_mul(a12, a12));
    const dfl dia = df_add(df_add(df_mul(b00, b00), df_mul(b11, b11)), df_mul(b22, b22));
    const dfl p2 = df_mul(df_add(dia, df_scale(off, 2.0f)), df_scale(third, 0.5f));
    *gap = p2.h >= 1e-26f ? 1.0f : 0.25f;
    if (!(p2.h >= 1e-26f)) return df_scale(q, is);   // all eigenvalues within 2e-13 of q (NaN: q is NaN)
    // y = 1 / sqrt(p2): FP32 estimate and one step from its exact residual
    const float y0 = rsqrtf(p2.h);
    const dfl u = df_mul(p2, df_two_prod(y0, y0));
    const float e = __fsub_rn(__fsub_rn(1.0f, u.h), u.l);
    const dfl y = df_fast_sum(y0, __fmul_rn(y0, __fmaf_rn(__fmul_rn(0.375f, e), e, __fmul_rn(0.5f, e))));
    const dfl p = df_mul(p2, y);
    b00 = df_mul(b00, y);
    b11 = df_mul(b11, y);
    b22 = df_mul(b22, y);
    const dfl c01 = df_mul(a01, y), c02 = df_mul(a02, y), c12 = df_mul(a12, y);
    const dfl m0 = df_sub(df_mul(b11, b22), df_mul(c12, c12));
    const dfl m1 = df_sub(df_mul(c01, b22), df_mul(c12, c02));
    const dfl m2 = df_sub(df_mul(c01, c12), df_mul(b11, c02));
    const dfl r = df_scale(df_add(df_sub(df_mul(b00, m0), df_mul(c01, m1)), df_mul(c02, m2)), 0.5f);
    const bool neg = r.h < 0.0f;
    dfl d = df_add(neg ? r : df_neg(r), 1.0f);
    if (d.h < 0.0f) d = {0.0f, 0.0f};   // |r| above 1 by rounding
    if (neg) *gap = d.h < 1e-9f ? 0.0f : sqrtf(d.h);
    // t in FP32 (two Newton steps from the start of its series), then one step in double-FP32
    const float c = d.h * (2.0f / 9.0f);
    float t0 = c * fmaf(2.0f / 3.0f, c, 1.0f);
#pragma unroll
    for (int it = 0; it < 2; ++it)
        t0 -= fmaf(t0, fmaf(t0, t0 - 6.0f, 9.0f), -2.0f * d.h) * __fdividef(1.0f, 3.0f * (1.0f - t0) * (3.0f - t0));
    const dfl v = df_mul(df_add(df_mul(df_two_sum(t0, -6.0f), t0), 9.0f), t0);
    const dfl res = df_sub(v, df_scale(d, 2.0f));
    const dfl t = df_two_sum(t0, -__fdividef(__fadd_rn(res.h, res.l), 3.0f * (1.0f - t0) * (3.0f - t0)));
    dfl beta;
    if (!neg) {
        beta = df_add(df_neg(t), 2.0f);
    } else {
        const dfl z = df_mul(df_mul(t, 3.0f), df_add(df_neg(t), 4.0f));
        beta = df_scale(df_add(df_add(df_neg(t), 2.0f), df_sqrt(z)), 0.5f);
    }
    return df_scale(df_add(q, df_mul(p, beta)), is);
}

// ln(x): near 1 as log1p of x - 1 (relative accuracy where the FTLE is near 0), else log of x
__device__ __forceinline__ float df_log(dfl x)
{
    const float d = __fadd_rn(__fsub_rn(x.h, 1.0f), x.l);
    return fabsf(d) < 0.5f ? log1pf(d) : logf(x.h);
}
