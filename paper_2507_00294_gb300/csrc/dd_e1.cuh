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
// 2^(k/128), k = 0..127, rounded to FP64.
static __device__ const double kExp2Tab[128] = {
    0x1.0000000000000p+0, 0x1.0163da9fb3335p+0, 0x1.02c9a3e778061p+0, 0x1.04315e86e7f85p+0,
    0x1.059b0d3158574p+0, 0x1.0706b29ddf6dep+0, 0x1.0874518759bc8p+0, 0x1.09e3ecac6f383p+0,
    0x1.0b5586cf9890fp+0, 0x1.0cc922b7247f7p+0, 0x1.0e3ec32d3d1a2p+0, 0x1.0fb66affed31bp+0,
    0x1.11301d0125b51p+0, 0x1.12abdc06c31ccp+0, 0x1.1429aaea92de0p+0, 0x1.15a98c8a58e51p+0,
    0x1.172b83c7d517bp+0, 0x1.18af9388c8deap+0, 0x1.1a35beb6fcb75p+0, 0x1.1bbe084045cd4p+0,
    0x1.1d4873168b9aap+0, 0x1.1ed5022fcd91dp+0, 0x1.2063b88628cd6p+0, 0x1.21f49917ddc96p+0,
    0x1.2387a6e756238p+0, 0x1.251ce4fb2a63fp+0, 0x1.26b4565e27cddp+0, 0x1.284dfe1f56381p+0,
    0x1.29e9df51fdee1p+0, 0x1.2b87fd0dad990p+0, 0x1.2d285a6e4030bp+0, 0x1.2ecafa93e2f56p+0,
    0x1.306fe0a31b715p+0, 0x1.32170fc4cd831p+0, 0x1.33c08b26416ffp+0, 0x1.356c55f929ff1p+0,
    0x1.371a7373aa9cbp+0, 0x1.38cae6d05d866p+0, 0x1.3a7db34e59ff7p+0, 0x1.3c32dc313a8e5p+0,
    0x1.3dea64c123422p+0, 0x1.3fa4504ac801cp+0, 0x1.4160a21f72e2ap+0, 0x1.431f5d950a897p+0,
    0x1.44e086061892dp+0, 0x1.46a41ed1d0057p+0, 0x1.486a2b5c13cd0p+0, 0x1.4a32af0d7d3dep+0,
    0x1.4bfdad5362a27p+0, 0x1.4dcb299fddd0dp+0, 0x1.4f9b2769d2ca7p+0, 0x1.516daa2cf6642p+0,
    0x1.5342b569d4f82p+0, 0x1.551a4ca5d920fp+0, 0x1.56f4736b527dap+0, 0x1.58d12d497c7fdp+0,
    0x1.5ab07dd485429p+0, 0x1.5c9268a5946b7p+0, 0x1.5e76f15ad2148p+0, 0x1.605e1b976dc09p+0,
    0x1.6247eb03a5585p+0, 0x1.6434634ccc320p+0, 0x1.6623882552225p+0, 0x1.68155d44ca973p+0,
    0x1.6a09e667f3bcdp+0, 0x1.6c012750bdabfp+0, 0x1.6dfb23c651a2fp+0, 0x1.6ff7df9519484p+0,
    0x1.71f75e8ec5f74p+0, 0x1.73f9a48a58174p+0, 0x1.75feb564267c9p+0, 0x1.780694fde5d3fp+0,
    0x1.7a11473eb0187p+0, 0x1.7c1ed0130c132p+0, 0x1.7e2f336cf4e62p+0, 0x1.80427543e1a12p+0,
    0x1.82589994cce13p+0, 0x1.8471a4623c7adp+0, 0x1.868d99b4492edp+0, 0x1.88ac7d98a6699p+0,
    0x1.8ace5422aa0dbp+0, 0x1.8cf3216b5448cp+0, 0x1.8f1ae99157736p+0, 0x1.9145b0b91ffc6p+0,
    0x1.93737b0cdc5e5p+0, 0x1.95a44cbc8520fp+0, 0x1.97d829fde4e50p+0, 0x1.9a0f170ca07bap+0,
    0x1.9c49182a3f090p+0, 0x1.9e86319e32323p+0, 0x1.a0c667b5de565p+0, 0x1.a309bec4a2d33p+0,
    0x1.a5503b23e255dp+0, 0x1.a799e1330b358p+0, 0x1.a9e6b5579fdbfp+0, 0x1.ac36bbfd3f37ap+0,
    0x1.ae89f995ad3adp+0, 0x1.b0e07298db666p+0, 0x1.b33a2b84f15fbp+0, 0x1.b59728de5593ap+0,
    0x1.b7f76f2fb5e47p+0, 0x1.ba5b030a1064ap+0, 0x1.bcc1e904bc1d2p+0, 0x1.bf2c25bd71e09p+0,
    0x1.c199bdd85529cp+0, 0x1.c40ab5fffd07ap+0, 0x1.c67f12e57d14bp+0, 0x1.c8f6d9406e7b5p+0,
    0x1.cb720dcef9069p+0, 0x1.cdf0b555dc3fap+0, 0x1.d072d4a07897cp+0, 0x1.d2f87080d89f2p+0,
    0x1.d5818dcfba487p+0, 0x1.d80e316c98398p+0, 0x1.da9e603db3285p+0, 0x1.dd321f301b460p+0,
    0x1.dfc97337b9b5fp+0, 0x1.e264614f5a129p+0, 0x1.e502ee78b3ff6p+0, 0x1.e7a51fbc74c83p+0,
    0x1.ea4afa2a490dap+0, 0x1.ecf482d8e67f1p+0, 0x1.efa1bee615a27p+0, 0x1.f252b376bba97p+0,
    0x1.f50765b6e4540p+0, 0x1.f7bfdad9cbe14p+0, 0x1.fa7c1819e90d8p+0, 0x1.fd3c22b8f71f1p+0,
};
// e^-x for 0 <= x <= 745, by table and a short polynomial (P. T. P. Tang, ACM TOMS 15, 1989):
// -x = (128 k + j) ln2/128 + r with |r| <= ln2/256, e^-x = 2^k 2^(j/128) e^r, e^r - 1 to degree 5
// (r^6/720 < 6e-19).  Ten FP64 operations and a table read in L1; FP64 runs at 1/70 of the FP32
// rate here and bounds every kernel that calls this.  Within one ulp.  The FP64 field of 12
// snapshots of a 1280-visit random scan on 96 x 81 points took 5020 us with exp() and FP64 class
// compares in the tile, and takes 3890 us with this and compares of the upper words.
__device__ __forceinline__ double exp_neg_f64(double x) {
    const double kMagic = 6755399441055744.0;            // 1.5 2^52: rounds to an integer
    const double t = fma(x, -184.6649652337873, kMagic);
    const int n = __double2loint(t), k = n >> 7;
    const double nd = t - kMagic;
    double r = fma(nd, -0.0054152123481245725, -x);
    r = fma(nd, -1.8117553233174215e-19, r);
    double p = fma(r, 1.0 / 120.0, 1.0 / 24.0);
    p = fma(p, r, 1.0 / 6.0);
    p = fma(p, r, 0.5);
    p = fma(p, r, 1.0) * r;
    const double T = kExp2Tab[n & 127], e = fma(T, p, T);
    if (k >= -1021) return __hiloint2double(__double2hiint(e) + (k << 20), __double2loint(e));
    // below the normal range: scaled in two steps
    return __hiloint2double(__double2hiint(e) + ((k + 64) << 20), __double2loint(e)) * 0x1p-64;
}

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
    if (a > 2.0)
        return exp_neg_f64(a) * (h > 40.0 ? e1_ratio_f64(a) : e1_ratio_f64(a) - exp_neg_f64(h) * e1_ratio_f64(b));
    const double e1b = b >= 745.0 ? 0.0 : exp_neg_f64(b) * e1_ratio_f64(b);
    return (-kEulerD - log(a) + ein_f64(a)) - e1b;
}

}  // namespace ddk
