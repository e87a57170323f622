// Standard normal quantile Phi^-1(p) for the Gaussian part of Alg. 1.
//
// Our own approximation, written from the relation
// Phi^-1(p) = sqrt(2) erfinv(2p - 1) and the split of erfinv used by Giles
// ("Approximating the erfinv function", GPU Computing Gems, 2010): with
// x = 2p - 1 and w = -ln(1 - x^2) = -ln(4 p (1 - p)),
//   erfinv(x) = x P1(w)          for w < 5   (p in (0.0017, 0.9983))
//   erfinv(x) = x P2(sqrt(w))    otherwise.
// Here the logarithm is taken in base 2, w2 = -log2(4p - 4p^2) = w / ln 2
// (the hardware lg2, no conversion), and the factor sqrt(2) is part of the
// polynomials: Phi^-1(p) = x Q1(w2 - c1) for w2 < 5 / ln 2, else
// x Q2(sqrt(w2) - c2), Q1 and Q2 of degree 9 with coefficients fitted for
// this library by weighted least squares against the exact quantile, for
// p in [2^-25, 1 - 2^-25].  There are two forms of the logarithm's argument, each
// one fused multiply-add:
//   4p - 4p^2  for any p (normal_quantile): accurate where x = 2p - 1 rounds;
//   1 - x^2    for the uniforms the hash produces, p = (2m + 1) 2^-24
//              (hash_quantile, hash_quantile2): x is exact in FP32 there, so both
//              round the same number, and this one is an operation shorter.
// lg2's error moves Q1 by less than 3e-8 relative; on those uniforms the result
// stays within 2.5e-7 relative (4.2e-8 absolute for |z| < 1/4) of the exact
// quantile.  Below 2^-25 Q2 is extrapolated (1e-6 relative at p = 1e-8, 3e-4 at
// 1e-10).
#pragma once

namespace glint {

// Phi^-1(p) from x = 2p - 1 and v = 4p (1 - p) = 1 - x^2.
__device__ __forceinline__ float quantile_of(float x, float v) {
    float w2;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(w2) : "f"(v));
    w2 = -w2;
    float P;
    if (w2 < 7.213475227f) {
        const float t = w2 - 3.606737614f;
        P = -4.593011249e-10f;
        P = fmaf(P, t, 1.750330991e-09f);
        P = fmaf(P, t, 5.068341480e-08f);
        P = fmaf(P, t, -5.430951546e-07f);
        P = fmaf(P, t, -1.123125344e-06f);
        P = fmaf(P, t, 7.127850404e-05f);
        P = fmaf(P, t, -5.900012329e-04f);
        P = fmaf(P, t, -2.838380402e-03f);
        P = fmaf(P, t, 2.417711467e-01f);
        P = fmaf(P, t, 2.123313427e+00f);
    } else {
        float r;
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(w2));
        const float t = r - 3.603367329f;
        P = 3.712571197e-05f;
        P = fmaf(P, t, -1.050955761e-04f);
        P = fmaf(P, t, -3.455006663e-05f);
        P = fmaf(P, t, 7.061248762e-04f);
        P = fmaf(P, t, -2.025795635e-03f);
        P = fmaf(P, t, 3.860775614e-03f);
        P = fmaf(P, t, -6.235580891e-03f);
        P = fmaf(P, t, 9.259297512e-03f);
        P = fmaf(P, t, 1.179382324e+00f);
        P = fmaf(P, t, 4.006434441e+00f);
    }
    return P * x;
}

// Any p in (0, 1).
__device__ __forceinline__ float normal_quantile(float p) {
    const float p4 = 4.f * p;
    return quantile_of(2.f * p - 1.f, fmaf(-p4, p, p4));
}

// p = (2m + 1) 2^-24, a uniform of the hash: normal_quantile's result.
__device__ __forceinline__ float hash_quantile(float p) {
    const float x = 2.f * p - 1.f;
    return quantile_of(x, fmaf(-x, x, 1.f));
}

// hash_quantile of two arguments in packed FP32, the same results.  The tail
// (0.35% of the uniforms) is evaluated for both when either needs it.
__device__ __forceinline__ f32x2 hash_quantile2(f32x2 p) {
    const f32x2 x = fma2(pack2(2.f, 2.f), p, pack2(-1.f, -1.f));
    const f32x2 v = fma2(mul2(x, pack2(-1.f, -1.f)), x, pack2(1.f, 1.f));
    float wa, wb;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(wa) : "f"(lo2(v)));
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(wb) : "f"(hi2(v)));
    const f32x2 t = sub2(pack2(-3.606737614f, -3.606737614f), pack2(wa, wb));
    f32x2 P = pack2(-4.593011249e-10f, -4.593011249e-10f);
    P = fma2(P, t, pack2(1.750330991e-09f, 1.750330991e-09f));
    P = fma2(P, t, pack2(5.068341480e-08f, 5.068341480e-08f));
    P = fma2(P, t, pack2(-5.430951546e-07f, -5.430951546e-07f));
    P = fma2(P, t, pack2(-1.123125344e-06f, -1.123125344e-06f));
    P = fma2(P, t, pack2(7.127850404e-05f, 7.127850404e-05f));
    P = fma2(P, t, pack2(-5.900012329e-04f, -5.900012329e-04f));
    P = fma2(P, t, pack2(-2.838380402e-03f, -2.838380402e-03f));
    P = fma2(P, t, pack2(2.417711467e-01f, 2.417711467e-01f));
    P = fma2(P, t, pack2(2.123313427e+00f, 2.123313427e+00f));
    if (fminf(wa, wb) <= -7.213475227f) {
        float ra, rb;
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(ra) : "f"(-wa));
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(rb) : "f"(-wb));
        const f32x2 s = add2(pack2(ra, rb), pack2(-3.603367329f, -3.603367329f));
        f32x2 Q = pack2(3.712571197e-05f, 3.712571197e-05f);
        Q = fma2(Q, s, pack2(-1.050955761e-04f, -1.050955761e-04f));
        Q = fma2(Q, s, pack2(-3.455006663e-05f, -3.455006663e-05f));
        Q = fma2(Q, s, pack2(7.061248762e-04f, 7.061248762e-04f));
        Q = fma2(Q, s, pack2(-2.025795635e-03f, -2.025795635e-03f));
        Q = fma2(Q, s, pack2(3.860775614e-03f, 3.860775614e-03f));
        Q = fma2(Q, s, pack2(-6.235580891e-03f, -6.235580891e-03f));
        Q = fma2(Q, s, pack2(9.259297512e-03f, 9.259297512e-03f));
        Q = fma2(Q, s, pack2(1.179382324e+00f, 1.179382324e+00f));
        Q = fma2(Q, s, pack2(4.006434441e+00f, 4.006434441e+00f));
        P = pack2(wa <= -7.213475227f ? lo2(Q) : lo2(P), wb <= -7.213475227f ? hi2(Q) : hi2(P));
    }
    return mul2(P, x);
}

}  // namespace glint
