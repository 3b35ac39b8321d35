// sigmoid.cuh -- the sigmoid of the formation (App. C.1 positions, opacities),
// each result rounded to FP32 once.
#pragma once

namespace gi {
namespace {

// 2^(j / 32), j = -16 .. 16, as sums of two floats.
__device__ const float2 kExp2Tab[33] = {
    {0.7071067690849304f, 1.2101617485882343e-08f}, {0.7225903868675232f, 1.662099968768871e-08f}, {0.7384130954742432f, -2.250449426810519e-08f},
    {0.7545822262763977f, -1.2479686617439256e-08f}, {0.7711054086685181f, 4.035452416673024e-09f}, {0.7879904508590698f, -2.830512713103417e-08f},
    {0.8052451610565186f, 4.918108587048664e-09f}, {0.8228777647018433f, -2.5624860455764065e-08f}, {0.8408964276313782f, -1.2377663338725142e-08f},
    {0.8593096733093262f, -2.4248087981959543e-08f}, {0.8781260848045349f, -4.617885185353998e-09f}, {0.8973545432090759f, -5.707522454656555e-09f},
    {0.9170040488243103f, -5.619638976384067e-09f}, {0.9370838403701782f, -2.331502813035513e-08f}, {0.9576032757759094f, 4.922664054163306e-09f},
    {0.9785720705986023f, -8.510902205216553e-09f}, {1.0f, 0.0f}, {1.0218971967697144f, -4.811559861650494e-08f},
    {1.0442737340927124f, 4.8334701574503924e-08f}, {1.0671404600143433f, -5.9337519786595294e-08f}, {1.0905077457427979f, -1.3077539939843064e-08f},
    {1.114386796951294f, -5.435540018083884e-08f}, {1.1387885808944702f, 5.386222312608879e-08f}, {1.1637248992919922f, -4.051441493402308e-08f},
    {1.1892070770263672f, 3.797635272917432e-08f}, {1.215247392654419f, -3.267394887984665e-08f}, {1.2418577671051025f, 4.496838101886169e-08f},
    {1.2690509557724f, 1.419333317542737e-09f}, {1.2968395948410034f, -4.018999533172973e-08f}, {1.3252366781234741f, -3.496373324196611e-08f},
    {1.3542555570602417f, -1.0123349269974824e-08f}, {1.3839099407196045f, -5.875577357983275e-08f}, {1.4142135381698608f, 2.4203234971764687e-08f},
};

// 1 / (1 + exp(-t)) as hi + lo, hi the nearest float: the App. C.1 positions
// ((tanh x + 1) / 2 = sigmoid(2 x)) and the opacities, in double-float
// arithmetic (Dekker 1971; Knuth, TAOCP 2, 4.2.2) on the FP32 units instead of
// FP64, whose rate on this part made it over half of the formation of a
// paper-mode step (step 110.8 -> 107.1 us at 768x512 / 70,000). With
// a = |t|: a log2(e) = n / 32 + f (n whole), exp(-a) = 2^(-n / 32) exp(-f ln 2)
// from the table and the exponential series to the fifth power (|f ln 2| <
// 0.011), then one Newton quotient. Relative error, measured against 64-bit
// mantissas on 10^8 values a range: at most 2^-42.6 for |t| <= 5, 2^-42.3 for
// t >= kSigmoidMin (2^-41.8 down to -60: a factor of 1.8 below what round_once
// allows, here 2.5). +infinity gives 1, NaN gives NaN.
constexpr float kSigmoidMin = -24.f;
__device__ __forceinline__ void sigmoid_dd(float t, float& hi, float& lo) {
    const float a = fminf(fabsf(t), 80.f);
    const float p = __fmul_rn(a, 1.442695f);  // log2(e) = 1.442695f + 1.925963e-08f
    const float pe = __fmaf_rn(a, 1.925963e-08f, __fmaf_rn(a, 1.442695f, -p));
    const float n = rintf(__fmul_rn(p, 32.f));
    const float fh = __fmaf_rn(n, -0.03125f, p);  // exact
    const float f = __fadd_rn(fh, pe), fl = __fadd_rn(__fsub_rn(fh, f), pe);
    // z = -f ln 2, ln 2 = 0.6931472f - 1.9046542e-09f
    const float zp = __fmul_rn(f, 0.6931472f);
    const float zh = -zp;
    const float zl = -__fadd_rn(__fmaf_rn(f, 0.6931472f, -zp), __fmaf_rn(f, -1.9046542e-09f, __fmul_rn(fl, 0.6931472f)));
    const int ni = __float2int_rn(n), k = (ni + 16) >> 5;
    const float2 T = kExp2Tab[16 - (ni - 32 * k)];  // 2^(-(n mod 32) / 32)
    // exp(z) - 1 = z + z^2 / 2 + z^3 (1/6 + z / 24 + z^2 / 120)
    const float q = __fmul_rn(zh, zh);
    const float ql = __fmaf_rn(__fmul_rn(2.f, zh), zl, __fmaf_rn(zh, zh, -q));
    const float tail = __fmul_rn(__fmul_rn(q, zh), __fmaf_rn(zh, __fmaf_rn(zh, 1.f / 120.f, 1.f / 24.f), 1.f / 6.f));
    const float h = __fmul_rn(0.5f, q);
    const float A = __fadd_rn(zh, h), ae = __fadd_rn(__fsub_rn(zh, A), h);
    const float e1 = __fadd_rn(__fadd_rn(__fmaf_rn(0.5f, ql, zl), ae), tail);
    // exp(-a) = 2^-k T (1 + A + e1)
    const float m = __fmul_rn(T.x, A), me = __fmaf_rn(T.x, A, -m);
    float eh = __fadd_rn(T.x, m);
    float el = __fadd_rn(__fsub_rn(T.x, eh), m);
    el = __fadd_rn(el, __fadd_rn(me, __fadd_rn(__fmaf_rn(T.x, e1, T.y), __fmul_rn(T.y, A))));
    const float sc = __int_as_float((127 - k) << 23);
    eh = __fmul_rn(eh, sc);
    el = __fmul_rn(el, sc);
    // (t < 0 ? exp(-a) : 1) / (1 + exp(-a))
    const float d = __fadd_rn(1.f, eh), dl = __fadd_rn(__fadd_rn(__fsub_rn(1.f, d), eh), el);
    const float nh = t < 0.f ? eh : 1.f, nl = t < 0.f ? el : 0.f;
    const float r = __frcp_rn(d);
    const float q0 = __fmul_rn(nh, r);
    const float rem = __fadd_rn(__fmaf_rn(-q0, d, nh), __fsub_rn(nl, __fmul_rn(q0, dl)));
    const float q1 = __fmul_rn(rem, r);
    hi = __fadd_rn(q0, q1);
    lo = __fadd_rn(__fsub_rn(q0, hi), q1);
    if (t != t) hi = t;
}

// The same in FP64, for the few values that need it (inlined: as a call it
// costs the step 1.4 us, inlined nothing measurable).
__device__ __forceinline__ double sigmoid_fp64(double t) {
    const double e = exp(-fabs(t));
    return (t < 0.0 ? e : 1.0) / (1.0 + e);
}

// m + e rounded once. ok: no value within 2^-41 of it (sigmoid_dd's error and
// the product's) rounds otherwise, that is, e is not that close to half a unit
// of m (Ziv, ACM TOMS 17, 1991): one value in 2^16 is not decided.
__device__ __forceinline__ float round_once(float m, float e, bool& ok) {
    const float r = __fadd_rn(m, e), rest = __fadd_rn(__fsub_rn(m, r), e);
    ok = __fmaf_rn(rest, 1.f + 0x1p-16f, r) == r;
    return r;
}

// sigmoid(t) rounded once, as FP64 rounds it.
__device__ __forceinline__ float opacity_of(float t) {
    float hi, lo;
    sigmoid_dd(t, hi, lo);
    bool ok;
    const float o = round_once(hi, lo, ok);
    return ok && t >= kSigmoidMin ? o : (float)sigmoid_fp64((double)t);
}

// size * sigmoid(2 x), rounded once (size = 0 .. 2^31 - 1, split into two
// floats, the first rounded towards zero so that it is a whole number in range).
__device__ __forceinline__ float raw_position(float x, int size) {
    const float t = __fmul_rn(2.f, x);
    float hi, lo;
    sigmoid_dd(t, hi, lo);
    const float sh = __int2float_rz(size), sl = (float)(size - (int)sh);
    const float m = __fmul_rn(hi, sh);
    bool ok;
    const float p = round_once(m, __fmaf_rn(lo, sh, __fmaf_rn(hi, sl, __fmaf_rn(hi, sh, -m))), ok);
    return ok && t >= kSigmoidMin ? p : (float)__dmul_rn(sigmoid_fp64(2.0 * (double)x), (double)size);
}

}  // namespace
}  // namespace gi
