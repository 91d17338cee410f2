// coef.cuh -- interpolation weights of one segment of the long-characteristic
// formal solution (voxel-node parabolic scheme R6 with series-stable
// evaluation R7), shared by the forward march and the adjoint march.
#pragma once

#include <cuda_runtime.h>

namespace rtk {

// 1/n! for n = 0..20
__device__ __forceinline__ double inv_fact(int n)
{
    const double f[21] = {1.0,
                          1.0,
                          1.0 / 2.0,
                          1.0 / 6.0,
                          1.0 / 24.0,
                          1.0 / 120.0,
                          1.0 / 720.0,
                          1.0 / 5040.0,
                          1.0 / 40320.0,
                          1.0 / 362880.0,
                          1.0 / 3628800.0,
                          1.0 / 39916800.0,
                          1.0 / 479001600.0,
                          1.0 / 6227020800.0,
                          1.0 / 87178291200.0,
                          1.0 / 1307674368000.0,
                          1.0 / 20922789888000.0,
                          1.0 / 355687428096000.0,
                          1.0 / 6402373705728000.0,
                          1.0 / 121645100408832000.0,
                          1.0 / 2432902008176640000.0};
    return f[n];
}

// 1 / q to about an ulp: the hardware's 20-bit estimate and one step of the third
// order Householder iteration for a reciprocal, r (1 + e + e^2) with e = 1 - q r
// (A. S. Householder, The Numerical Treatment of a Single Nonlinear Equation, 1970,
// ch. 4): three FP64 instructions where a correctly rounded division takes about
// ten.  Outside [2^-900, 2^900], where the estimate would leave the normal range:
// the division.
__device__ __forceinline__ bool rcp64_in_range(double q)
{
    return (((unsigned)__double2hiint(q) >> 20) & 0x7ffu) - 123u <= 1800u;
}
__device__ __forceinline__ double rcp64(double q)
{
    if (!rcp64_in_range(q)) return 1.0 / q;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(q));
    const double e = fma(-q, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// a / q to half an ulp or a little more: its residual corrects a rcp64(q).
__device__ __forceinline__ double div64(double a, double q)
{
    if (!rcp64_in_range(q)) return a / q;
    const double r = rcp64(q), t = a * r;
    return fma(fma(-t, q, a), r, t);
}

// x < 1 and x < 1/2 for x >= 0, from the high word: off the FP64 pipe (a NaN is neither).
__device__ __forceinline__ bool below_one(double x) { return (unsigned)__double2hiint(x) < 0x3ff00000u; }
__device__ __forceinline__ bool below_half(double x) { return (unsigned)__double2hiint(x) < 0x3fe00000u; }

// E below x = 1: 1 - e0, and from 1/2 on, where 1 - x is exact, x f1 + (1 - x); one FP64
// instruction on operands chosen off that pipe.
__device__ __forceinline__ double small_E(double x, double f1, double e0)
{
    const bool half = below_half(x);
    return fma(half ? -1.0 : x, half ? e0 : f1, half ? 1.0 : 1.0 - x);
}

// h1(x) = (e^{-x} - 1 + x) / x^2 and h2(x) = f2(x) / x^2 (see below) on [0, 1]:
// their values at 0 plus x times polynomials fitted to (h - h(0)) / x at Chebyshev
// nodes (fit error 1e-18 of h, under FP64 rounding).
__device__ __forceinline__ double h1_small(double x)
{
    double h = 7.722609696190044e-12;
    h = fma(h, x, -1.514301957269351e-10);
    h = fma(h, x, 2.0743464091464554e-09);
    h = fma(h, x, -2.5039626817896517e-08);
    h = fma(h, x, 2.755654152433202e-07);
    h = fma(h, x, -2.7557286761537225e-06);
    h = fma(h, x, 2.480158640720805e-05);
    h = fma(h, x, -0.00019841269825620665);
    h = fma(h, x, 0.001388888888872712);
    h = fma(h, x, -0.00833333333333247);
    h = fma(h, x, 0.04166666666666665);
    h = fma(h, x, -0.16666666666666666);
    return fma(h, x, 0.5);
}
__device__ __forceinline__ double h2_small(double x)
{
    double h = 6.667117678494612e-12;
    h = fma(h, x, -1.2965202422838241e-10);
    h = fma(h, x, 1.754862018413882e-09);
    h = fma(h, x, -2.086586606418334e-08);
    h = fma(h, x, 2.2546219039428151e-07);
    h = fma(h, x, -2.204582705953453e-06);
    h = fma(h, x, 1.9290122676595323e-05);
    h = fma(h, x, -0.00014880952367301683);
    h = fma(h, x, 0.0009920634920493816);
    h = fma(h, x, -0.005555555555554801);
    h = fma(h, x, 0.024999999999999984);
    h = fma(h, x, -0.08333333333333333);
    return fma(h, x, 1.0 / 6.0);
}

// Weights of one segment of optical depth x followed by p.
//   e0 = 1 - e^{-x},  f1 = (x - e0)/x,  f2 = (x(2 - e0) - 2 e0)/x = 2 f1 - e0
//   parabolic: alpha = e0 - f1 - f2/(x+p), beta = f1 + f2/p, gamma = -x f2/(p (x+p))
//   linear:    alpha = e0 - f1,           beta = f1,         gamma = 0
// f1 and f2 cancel catastrophically when evaluated from e0 at small x; below 1
// they come from polynomials, above it from the exponential.  The three quotients
// of the parabola share one.  The FP64 pipe bounds every kernel that
// evaluates these: about 44 instructions of it for a small x and for a large one
// (62 and 80 with the 19-term series, expm1 and divisions of Coef64Series).  Mean
// errors of E, alpha, beta, gamma in half ulps of their terms, Coef64Series -> here:
// below 0.5 0.27, 0.28, 0.49, 0.77 -> 0.27, 0.29, 0.50, 0.69; in [0.5, 1] 0.57, 0.74,
// 1.58, 11.0 -> 0.46, 0.38, 0.56, 0.70; in [1, 4] 3.2, 0.37, 0.69, 2.51 -> 0.38, 0.40,
// 0.73, 2.51; above, E keeps its relative accuracy, 0.18, 0.39, 0.67 -> 0.18, 0.40, 0.72.
struct Coef64 {
    __device__ __forceinline__ static void eval(double x, double p, bool para, double &E, double &al, double &be,
                                                double &ga)
    {
        double e0, f1, f2;
        if (below_one(x)) {
            f1 = x * h1_small(x);
            f2 = (x * x) * h2_small(x);
            e0 = fma(-x, f1, x);
            E = small_E(x, f1, e0);
        } else {
            E = exp(-x);
            e0 = 1.0 - E;
            f1 = div64(x - e0, x);
            f2 = fma(2.0, f1, -e0);
        }
        al = e0 - f1;
        be = f1;
        ga = 0.0;
        if (para) {
            const double D = x + p, t = div64(f2, p * D);
            al = fma(-t, p, al);
            be = fma(t, D, be);
            ga = -(x * t);
        }
    }
};

// The same weights from 19-term series and expm1, each quotient divided: those
// of the nearest-neighbour operator, whose entries stay the same to the last bit
// (a line problem at eps_l = 1e-4 and chi_l / chi_c = 1e6 turns a change of their
// rounding into 1e-5 of its iterates).
struct Coef64Series {
    static constexpr int NS = 19;  // series terms for x < 0.5
    __device__ __forceinline__ static void eval(double x, double p, bool para, double &E, double &al, double &be,
                                                double &ga)
    {
        double e0, f1, f2;
        if (x < 0.5) {
            double h1 = 0.0, h2 = 0.0;
#pragma unroll
            for (int n = NS + 1; n >= 2; --n) h1 = inv_fact(n) - x * h1;        // sum (-x)^(n-2)/n!
#pragma unroll
            for (int m = NS + 1; m >= 3; --m) h2 = (double)(m - 2) * inv_fact(m) - x * h2;
            f1 = x * h1;
            f2 = (x * x) * h2;
            e0 = x - x * f1;
            E = 1.0 - e0;
        } else {
            double em = expm1(-x);
            e0 = -em;
            E = 1.0 + em;
            f1 = (x - e0) / x;
            f2 = (x * (2.0 - e0) - 2.0 * e0) / x;
        }
        if (para) {
            double iD = 1.0 / (x + p), ip = 1.0 / p;
            al = (e0 - f1) - f2 * iD;
            be = f1 + f2 * ip;
            ga = -(x * f2) * (ip * iD);
        } else {
            al = e0 - f1;
            be = f1;
            ga = 0.0;
        }
    }
};

// FP32 weights for the marches that evaluate them per segment (batch members,
// the full FP32 formal solution, chunked sweeps).  Below x = 1, f1 = x h1(x)
// and f2 = x^2 h2(x) with h1(x) = (e^{-x} - 1 + x)/x^2 = 1/2 - x/6 + x^2/24 - ...
// and h2(x) = f2(x)/x^2 = 1/6 - x/12 + x^2/40 - ... taken from degree-6
// polynomials fitted to those definitions on [0, 1] in the minimax sense of
// relative error (fit error 5e-10 for h1, 1.4e-9 for h2, under FP32 rounding);
// above, from the exponential as in Coef64.  Reciprocals are the hardware
// approximation (about one ulp), ample for FP32 weights.
struct Coef32 {
    __device__ __forceinline__ static float h1(float x)
    {
        float h = 1.687989424681291e-05f;
        h = fmaf(h, x, -1.8817881937138736e-04f);
        h = fmaf(h, x, 1.3820757158100605e-03f);
        h = fmaf(h, x, -8.330963551998138e-03f);
        h = fmaf(h, x, 4.1666269302368164e-02f);
        h = fmaf(h, x, -1.66666641831398e-01f);
        return fmaf(h, x, 0.5f);
    }
    __device__ __forceinline__ static float h2(float x)
    {
        float h = 1.2951083590451162e-05f;
        h = fmaf(h, x, -1.4058091619517654e-04f);
        h = fmaf(h, x, 9.86545579507947e-04f);
        h = fmaf(h, x, -5.553617607802153e-03f);
        h = fmaf(h, x, 2.4999670684337616e-02f);
        h = fmaf(h, x, -8.333331346511841e-02f);
        return fmaf(h, x, 1.666666716337204e-01f);
    }
    __device__ __forceinline__ static float rcp(float v) { return __fdividef(1.0f, v); }
    __device__ __forceinline__ static void eval(float x, float p, bool para, float &E, float &al, float &be, float &ga)
    {
        float e0, f1, f2;
        if (x < 1.0f) {
            f1 = x * h1(x);
            f2 = (x * x) * h2(x);
            e0 = x - x * f1;
            E = 1.0f - e0;
        } else {
            E = __expf(-x);
            e0 = 1.0f - E;
            const float ix = rcp(x);
            f1 = (x - e0) * ix;
            f2 = (x * (2.0f - e0) - 2.0f * e0) * ix;
        }
        if (para) {
            const float iD = rcp(x + p), ip = rcp(p);
            al = (e0 - f1) - f2 * iD;
            be = f1 + f2 * ip;
            ga = -(x * f2) * (ip * iD);
        } else {
            al = e0 - f1;
            be = f1;
            ga = 0.0f;
        }
    }
};

// Derivatives of (E, alpha, beta, gamma) with respect to x = dtau_k and
// p = dtau_{k+1}, from  e0' = E, f1' = (e0 - f1)/x = g1, f2' = e0 - f1 - f2/x = g2
// (below 1 their power series, 19 terms: 1 - h1 - x h1 loses up to half the bits of an ulp more):
//   parabolic: alpha = e0 - f1 - f2/(x+p), beta = f1 + f2/p, gamma = -x f2/(p (x+p))
//   linear:    alpha = e0 - f1,           beta = f1
struct Coef64D {
    __device__ __forceinline__ static void eval(double x, double p, bool para, double &E, double &al, double &be,
                                                double &ga, double &dE, double &dal_x, double &dbe_x, double &dga_x,
                                                double &dal_p, double &dbe_p, double &dga_p)
    {
        double e0, f1, f2, g1, g2;
        if (below_one(x)) {
            constexpr int NS = 19;
            double k1 = 0.0, k2 = 0.0;
            // g1 = sum_{n>=2} (-1)^n (n-1) x^(n-2) / n!,  g2 = sum_{m>=3} (-1)^(m+1) (m-2)(m-1) x^(m-2) / m!
#pragma unroll
            for (int n = NS + 1; n >= 2; --n) k1 = fma(-x, k1, (double)(n - 1) * inv_fact(n));
#pragma unroll
            for (int m = NS + 1; m >= 3; --m) k2 = fma(-x, k2, (double)((m - 2) * (m - 1)) * inv_fact(m));
            f1 = x * h1_small(x);
            f2 = (x * x) * h2_small(x);
            e0 = fma(-x, f1, x);
            E = small_E(x, f1, e0);
            g1 = k1;
            g2 = x * k2;
        } else {
            E = exp(-x);
            e0 = 1.0 - E;
            f1 = div64(x - e0, x);
            f2 = fma(2.0, f1, -e0);
            g1 = div64(e0 - f1, x);
            g2 = (e0 - f1) - div64(f2, x);
        }
        dE = -E;
        if (para) {
            const double D = x + p, iD = 1.0 / D, ip = 1.0 / p;
            al = (e0 - f1) - f2 * iD;
            be = f1 + f2 * ip;
            ga = -(x * f2) * (ip * iD);
            dal_x = E - g1 - g2 * iD + f2 * iD * iD;
            dal_p = f2 * iD * iD;
            dbe_x = g1 + g2 * ip;
            dbe_p = -f2 * ip * ip;
            dga_x = -(f2 * p + x * g2 * D) * (ip * iD * iD);
            dga_p = x * f2 * (x + 2.0 * p) * (ip * ip * iD * iD);
        } else {
            al = e0 - f1;
            be = f1;
            ga = 0.0;
            dal_x = E - g1;
            dbe_x = g1;
            dga_x = 0.0;
            dal_p = dbe_p = dga_p = 0.0;
        }
    }
};

}  // namespace rtk
