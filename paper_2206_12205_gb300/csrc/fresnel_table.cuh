// Piecewise polynomials of the auxiliary function G of the Fresnel integrals, for the FP64
// evaluation of K5:  F(s) = C(s) + i S(s) = sgn(s) ((1+i)/2 - G(|s|) exp(i pi s^2 / 2)).
//
// F' = exp(i pi x^2 / 2) gives the differential equation G' = -1 - i pi x G, G(0) = (1+i)/2, from which
// everything below follows; G is smooth and falls like i/(pi x).  A polynomial of degree 9 per
// interval takes 20 FP64 operations where the power series took 96 and the continued fraction up
// to 400, without the divergence between the two (GB300 runs FP64 at 1/64 of the FP32 rate, so
// operations are what the evaluation pays for).  Intervals:
//   x < 8:  128 of width 1/16.  Taylor coefficients about the centre a from the differential
//           equation, c_1 = -1 - i pi a c_0, (n+1) c_{n+1} = -i pi (a c_n + c_{n-1}), and c_0 = G(a) by
//           carrying the same expansion from centre to centre in double-double (the homogeneous
//           solution has modulus 1, so errors do not grow).  The first term left out is at most
//           (sqrt(pi/2)/32)^10 / 5! = 7e-17.
//   x >= 8: 16 per octave up to 2^11.  G = sum_k a_k x^-(2k+1), a_0 = i/pi, a_{k+1} = -i (2k+1) a_k / pi
//           (asymptotic; the terms left out are below 1e-18 at x = 8), expanded about the centre with the
//           binomial series; |x/a - 1| <= 1/32, so the first term left out is below 1e-16 of G.
// Built at compile time (constexpr), 40 KB.
#pragma once

#include <cuda_runtime.h>

namespace fdas {

constexpr int FRESNEL_TERMS = 10;        // coefficients per interval
constexpr int FRESNEL_UNIFORM = 128;     // intervals of width 1/16 below 8
constexpr int FRESNEL_INTERVALS = FRESNEL_UNIFORM + 8 * 16;

// Double-double arithmetic for the table (Dekker's product, Knuth's sum).
struct ct_dd {
    double h, l;
};
constexpr ct_dd dd_sum(double a, double b) {
    const double s = a + b, bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}
constexpr ct_dd dd_prod(double a, double b) {
    constexpr double K = 134217729.0;    // 2^27 + 1
    const double p = a * b;
    const double ta = K * a, ah = ta - (ta - a), al = a - ah;
    const double tb = K * b, bh = tb - (tb - b), bl = b - bh;
    return {p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
constexpr ct_dd operator+(ct_dd a, ct_dd b) {
    const ct_dd s = dd_sum(a.h, b.h);
    return dd_sum(s.h, s.l + a.l + b.l);
}
constexpr ct_dd operator*(ct_dd a, ct_dd b) {
    const ct_dd p = dd_prod(a.h, b.h);
    return dd_sum(p.h, p.l + (a.h * b.l + a.l * b.h));
}
constexpr ct_dd operator-(ct_dd a) { return {-a.h, -a.l}; }
constexpr ct_dd dd_over(ct_dd a, double n) {       // a / n: one correction step
    const double q = a.h / n;
    const ct_dd p = dd_prod(q, n);
    return dd_sum(q, (((a.h - p.h) - p.l) + a.l) / n);
}

struct FresnelTable {
    double c[FRESNEL_TERMS][FRESNEL_INTERVALS][2];     // [coefficient][interval] re, im

    constexpr FresnelTable() : c() {
        constexpr ct_dd PI = {3.141592653589793116, 1.2246467991473532e-16};
        constexpr int T = 16;                          // terms carried from centre to centre
        ct_dd re = {0.5, 0.0}, im = {0.5, 0.0};        // G at `from`
        double from = 0.0;
        for (int k = -1; k < FRESNEL_UNIFORM; k++) {
            // Taylor coefficients about `from`: (n+1) c_{n+1} = -delta_{n0} - i pi (a c_n + c_{n-1})
            ct_dd cr[T] = {}, ci[T] = {};
            cr[0] = re;
            ci[0] = im;
            for (int n = 0; n + 1 < T; n++) {
                ct_dd wr = ct_dd{from, 0.0} * cr[n], wi = ct_dd{from, 0.0} * ci[n];
                if (n > 0) {
                    wr = wr + cr[n - 1];
                    wi = wi + ci[n - 1];
                }
                wr = PI * wr;
                wi = PI * wi;
                cr[n + 1] = n == 0 ? wi + ct_dd{-1.0, 0.0} : dd_over(wi, n + 1);      // -i (wr + i wi) = wi - i wr
                ci[n + 1] = n == 0 ? -wr : dd_over(-wr, n + 1);
            }
            if (k >= 0)
                for (int n = 0; n < FRESNEL_TERMS; n++) {
                    c[n][k][0] = cr[n].h;
                    c[n][k][1] = ci[n].h;
                }
            const double to = (k + 1.5) / 16.0;
            const ct_dd u = {to - from, 0.0};
            re = cr[T - 1];
            im = ci[T - 1];
            for (int n = T - 2; n >= 0; n--) {
                re = re * u + cr[n];
                im = im * u + ci[n];
            }
            from = to;
        }
        constexpr double IPI = 0.31830988618379067154;
        for (int o = 0; o < 8; o++)
            for (int q = 0; q < 16; q++) {
                const double a = (double)(8 << o) * (1.0 + (q + 0.5) / 16.0);
                for (int n = 0; n < FRESNEL_TERMS; n++) {
                    double sr = 0.0, si = 0.0;
                    double term[14] = {};                 // |a_k| a^-(2k+1) times the binomial factor of u^n
                    double ak = IPI / a;
                    for (int k = 0; k < 14; k++) {
                        double b = ak;
                        for (int i = 0; i < n; i++) b *= -(2.0 * k + 1.0 + i) / ((i + 1.0) * a);
                        term[k] = b;
                        ak *= (2.0 * k + 1.0) * IPI / (a * a);
                    }
                    for (int k = 13; k >= 0; k--) {       // a_k = i (-i)^k |a_k|: i, 1, -i, -1, ...
                        const double v = (k & 2) ? -term[k] : term[k];
                        if (k & 1) sr += v; else si += v;
                    }
                    c[n][FRESNEL_UNIFORM + 16 * o + q][0] = sr;
                    c[n][FRESNEL_UNIFORM + 16 * o + q][1] = si;
                }
            }
    }
};

__device__ constexpr FresnelTable fresnel_table{};

// The interval of x in [0, 2^11) (a value a little outside an interval is as good) and its centre.
struct FresnelSpot {
    int idx;
    float centre;
};
__device__ __forceinline__ FresnelSpot fresnel_spot(float x) {
    if (x < 8.f) {
        const int i = (int)(x * 16.f);
        return {i, ((float)i + 0.5f) * 0.0625f};
    }
    const unsigned b = __float_as_uint(x);
    const float centre = __uint_as_float((b & 0xFFF80000u) | 0x00040000u);
    const int i = (int)(b >> 19) - (130 << 4);      // exponent 130: 8 <= x < 16
    return {FRESNEL_UNIFORM + (i < 127 ? i : 127), centre};
}

}  // namespace fdas
