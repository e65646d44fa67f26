// dd_e1.cuh -- device math for the E_1 difference of Eq. 1/2 (FP32 and FP64).
//
// E_1(v) = int_v^inf e^-u/u du (definition below Eq. 2).  Every pair term of the
// field is  E_1(a) - E_1(b)  with a = rho^2/w1 <= b = rho^2/w0.  Writing h = b - a and
// r = b/a - 1 = (w1 - w0)/w0, the substitution u = a(1 + r s) gives
//     E_1(a) - E_1(b) = e^-a int_0^1 r e^{-h s} / (1 + r s) ds = e^-a sum_m c_m h^m,
//     c_m = (-1)^m J_m(r) / m!,   J_m(r) = int_0^1 r s^m / (1 + r s) ds,
// an alternating series whose m-th term is bounded by ln(1+r) h^m / m!.  The c_m
// depend on the (visit, snapshot) pair only, so they are computed once in FP64
// (dd_field.cu) and the per-pair work is e^-a times a polynomial in h ("moment
// regime", used while h <= 1/2).  Larger h is rare (recent, nearby visits); there
// E_1(a) and E_1(b) are formed separately (the difference is then well conditioned,
// E_1(b) <= e^-h E_1(a)):  Ein series (A&S 5.1.11) below x = 1 (FP32) / 2 (FP64), a
// rational fit of x e^x E_1(x) (generated by gen_e1_constants.py) above.
#pragma once
#include <cuda_runtime.h>

namespace ddk {

constexpr float kLog2eF = 1.44269504088896340736f;
constexpr float kEulerF = 0.577215664901532860606f;
constexpr double kEulerD = 0.577215664901532860606512090082;

// ------------------------------------------------------------------ FP32 helpers
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float lg2_approx(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// e^-x with the rounding of x*log2(e) compensated (one extra FMA pair).
__device__ __forceinline__ float exp_neg_f32(float x) {
    float t = x * kLog2eF;
    float lo = fmaf(x, kLog2eF, -t) + x * 1.9259629911e-8f;   // log2(e) - fl32(log2(e))
    return ex2_approx(-t) * fmaf(-lo, 0.69314718056f, 1.0f);
}

// Ein(x) = sum_{k>=1} (-1)^{k+1} x^k / (k k!) for 0 <= x <= 1; 10 terms (truncation < 3e-9 x).
__device__ __forceinline__ float ein_f32(float x) {
    float p = -2.75573192239858909e-08f;
    p = fmaf(p, x, 3.06192435822065443e-07f);
    p = fmaf(p, x, -3.10019841269841270e-06f);
    p = fmaf(p, x, 2.83446712018140604e-05f);
    p = fmaf(p, x, -2.31481481481481490e-04f);
    p = fmaf(p, x, 1.66666666666666677e-03f);
    p = fmaf(p, x, -1.04166666666666661e-02f);
    p = fmaf(p, x, 5.55555555555555525e-02f);
    p = fmaf(p, x, -2.5e-01f);
    p = fmaf(p, x, 1.0f);
    return p * x;
}

// E_1(x) for x >= 1: e^-x P*(x) / (x Q*(x)); the rational in 1/x fits x e^x E_1(x)
// to 1.8e-8 relative on [1, inf) (gen_e1_constants.py).
__device__ __forceinline__ float e1_large_f32(float x) {
    float p = fmaf(fmaf(fmaf(fmaf(9.999999834e-01f, x, 8.553607022e+00f), x, 1.799050464e+01f), x,
                        8.602362612e+00f), x, 2.675161457e-01f);
    float q = fmaf(fmaf(fmaf(x + 9.553598517e+00f, x, 2.554479304e+01f), x, 2.101735711e+01f), x,
                   3.945961475e+00f);
    return exp_neg_f32(x) * p * rcp_approx(x * q);
}

// E_1(a) - E_1(b) for 1 <= a < 87, a <= b: e1_large_f32 of a and b at once, one f32x2
// instruction per step (each half rounds exactly as e1_large_f32 does); E_1(b) counts as 0
// from b = 87 on (below the FP32 normal range).
__device__ __forceinline__ float e1diff_large_pair_f32(float a, float b) {
    const float2 x = make_float2(a, b);
    auto c2 = [](float c) { return make_float2(c, c); };
    float2 p = __ffma2_rn(c2(9.999999834e-01f), x, c2(8.553607022e+00f));
    p = __ffma2_rn(p, x, c2(1.799050464e+01f));
    p = __ffma2_rn(p, x, c2(8.602362612e+00f));
    p = __ffma2_rn(p, x, c2(2.675161457e-01f));
    float2 q = __fadd2_rn(x, c2(9.553598517e+00f));
    q = __ffma2_rn(q, x, c2(2.554479304e+01f));
    q = __ffma2_rn(q, x, c2(2.101735711e+01f));
    q = __ffma2_rn(q, x, c2(3.945961475e+00f));
    // e^-x as in exp_neg_f32
    const float2 t = __fmul2_rn(x, c2(kLog2eF));
    const float2 lo = __ffma2_rn(x, c2(1.9259629911e-8f), __ffma2_rn(x, c2(kLog2eF), make_float2(-t.x, -t.y)));
    const float2 e = __fmul2_rn(make_float2(ex2_approx(-t.x), ex2_approx(-t.y)),
                                __ffma2_rn(make_float2(-lo.x, -lo.y), c2(0.69314718056f), c2(1.0f)));
    const float2 xq = __fmul2_rn(x, q);
    const float2 v = __fmul2_rn(__fmul2_rn(e, p), make_float2(rcp_approx(xq.x), rcp_approx(xq.y)));
    return b >= 87.0f ? v.x : v.x - v.y;
}

// E_1(a) - E_1(a + h) beyond the exponent series' range (general regime); ell = ln((a + h)/a).
static __device__ __forceinline__ float e1diff_general_f32(float a, float h, float ell) {
    const float b = a + h;
    if (b <= 1.0f) return ell - (ein_f32(b) - ein_f32(a));          // ln(b/a) - [Ein(b) - Ein(a)]
    if (a > 1.0f) return e1diff_large_pair_f32(a, b);
    const float e1b = b >= 87.0f ? 0.0f : e1_large_f32(b);
    const float e1a = -kEulerF - lg2_approx(a) * 0.69314718056f + ein_f32(a);
    return e1a - e1b;
}

// ------------------------------------------------------------------ FP64 helpers
static __device__ __constant__ double kEin64[30] = {
    1.00000000000000000e+00,
    -2.50000000000000000e-01,
    5.55555555555555525e-02,
    -1.04166666666666661e-02,
    1.66666666666666677e-03,
    -2.31481481481481490e-04,
    2.83446712018140604e-05,
    -3.10019841269841270e-06,
    3.06192435822065443e-07,
    -2.75573192239858909e-08,
    2.27746439867651998e-09,
    -1.73972974898900835e-10,
    1.23531106437089348e-11,
    -8.19338971266408865e-13,
    5.09810915454654461e-14,
    -2.98717333274211578e-15,
    1.65379838490912975e-16,
    -8.67733720477012532e-18,
    4.32665012980227901e-19,
    -2.05515881165608254e-20,
    9.32044812542441022e-22,
    -4.04399608747753346e-23,
    1.68181311766551469e-24,
    -6.71557321290049327e-26,
    2.57878011375378935e-27,
    -9.53690870471075953e-29,
    3.40136661622057234e-30,
    -1.17138901323922786e-31,
    3.89998720222335054e-33,
    -1.25666254293863529e-34
};

// Ein(x) for 0 <= x <= 2; 30 terms (truncation < 1e-24).
__device__ __forceinline__ double ein_f64(double x) {
    double p = kEin64[29];
#pragma unroll
    for (int k = 28; k >= 0; --k) p = fma(p, x, kEin64[k]);
    return p * x;
}

// x E_1(x) e^x for x > 2 as P*(x) / Q*(x): a rational of degree 9 in 1/x, within 3.8e-18
// relative on [2, inf) (gen_e1_constants.py); every coefficient is positive, so Horner's
// rounding stays at a few ulp.  e1_ratio_f64 returns E_1(x) e^x = P* / (x Q*): 19 FMAs and a
// division, where the continued fraction of A&S 5.1.22 took up to 60 steps of two divisions
// (one such term alone kept a warp busy for about 70 us).
static __device__ __constant__ double kE1P64[10] = {
    0.99999999999999999637, 41.073876422688601655, 645.56102424747329172, 4990.1513622650472973,
    20326.288895540010955,  43481.796815695771445, 45998.061135410915445, 20938.950545390477397,
    2973.7124827043992538,  32.248772351909912869};
static __device__ __constant__ double kE1Q64[10] = {
    1.0,                    42.073876422688585967, 685.63490067017287432, 5597.6385100868289719,
    24781.100863259999818,  60291.656989110476737, 78186.977491438231373, 49908.775676338818251,
    13308.241550527079719,  1001.6481696827983802};
__device__ __forceinline__ double e1_ratio_f64(double x) {
    double p = kE1P64[0], q = kE1Q64[0];
#pragma unroll
    for (int k = 1; k < 10; ++k) {
        p = fma(p, x, kE1P64[k]);
        q = fma(q, x, kE1Q64[k]);
    }
    return p / (x * q);
}

// E_1(a) - E_1(a + h) for h > 1/2 in FP64; ell = ln((a + h)/a).
static __device__ __noinline__ double e1diff_general_f64(double a, double h, double ell) {
    const double b = a + h;
    if (b <= 2.0) return ell - (ein_f64(b) - ein_f64(a));
    // E_1(b) <= e^-h E_1(a): below 5e-18 of the difference from h = 40 on
    if (a > 2.0) return exp(-a) * (h > 40.0 ? e1_ratio_f64(a) : e1_ratio_f64(a) - exp(-h) * e1_ratio_f64(b));
    const double e1b = b >= 745.0 ? 0.0 : exp(-b) * e1_ratio_f64(b);
    return (-kEulerD - log(a) + ein_f64(a)) - e1b;
}

}  // namespace ddk
