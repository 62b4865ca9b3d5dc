// K5: sub-bin refinement of f-z candidates by gradient ascent on the Fourier-interpolated power
// (the plane of Sec. 2.1 evaluated between its grid points; derivatives by the adjoint sums).
//
// A plane peak sits on the integer grid (r, z_i); the signal that made it lies in between.  With
// the plane's m-tap window anchored at bin k0, the interpolated amplitude and power are
//   A(r, z) = sum_{k = k0-m/2}^{k0+m/2-1} Xhat_k conj(I(k - r, z)),   P = |A|^2,
// where I(q, z) = M_0(q, z) is the unnormalised response of a constant-fdot sinusoid (z in bins of
// drift over the observation, Eq. fdotz) and M_p(q, z) = int_0^1 u^p exp(i pi (z u^2 - 2 q u)) du.
// Differentiating under the integral, dI(k - r, z)/dr = 2 pi i M_1 and dI/dz = i pi M_2, so
//   dP/dr = 2 Re(conj(A) sum_k Xhat_k conj(2 pi i M_1)),  dP/dz = 2 Re(conj(A) sum_k Xhat_k conj(i pi M_2)).
// One warp evaluates one point: lane l takes taps l, l + 32, ... (coalesced spectrum reads, and
// neighbouring lanes take neighbouring taps, which fall in the same branch below); the three sums
// are reduced with xor shuffles, after which every lane holds the same bits, so the ascent's
// control flow is warp-uniform.
//
// Moments of one tap, for z >= 0 (z < 0 through M_p(q, z) = conj(M_p(-q, -z))), v(u) = z u - q:
//  * far tap, min_{u in [0,1]} |v| >= c max(1, sqrt z): no stationary phase near [0, 1].  Repeated
//    integration by parts (dE/du = 2 pi i v E, E = exp(i pi (z u^2 - 2 q u))) gives, at each end,
//    with w = 1/(2 pi i v) and t = z/(2 pi i v^2):
//      M_0 = [E w S0]_0^1,  M_1 = [E (u w S0 - w^2 S1)]_0^1,  M_2 = [E (u^2 w S0 - 2 u w^2 S1 + 2 w^3 S2)]_0^1,
//      S0 = sum_k (2k-1)!! t^k,  S1 = sum_k (2k+1)!! t^k,  S2 = sum_k (k+1)(2k+1)!! t^k.
//    |t| <= 1/(2 pi c^2), so 5 terms (c = 6) leave a truncation below FP32 rounding and 7 terms
//    (c = 12) below 1e-14.
//  * near tap, z >= 1: the Fresnel form.  Completing the square, with F = C + iS written at each
//    end as F(s) = c + d exp(i pi s^2/2) (its power series for |s| <= 1.5, 2.5 in FP64, where
//    d = 0; otherwise c = sgn(s)(1+i)/2 and d = -sgn(s) G(|s|),
//    G(x) = (1+i)/(2 sqrt(pi)) K((sqrt(pi)/2)(1-i) x), K the Laplace continued fraction of
//    sqrt(pi) exp(w^2) erfc(w); its depth, set per lane, bounds the warp's time, hence the wider
//    series range in FP64),
//      sqrt(2z) M_0 = (c1 - c0) exp(-i pi q^2/z) + d1 exp(i pi (z - 2q)) - d0,
//      s0 = -q sqrt(2/z),  s1 = (z - q) sqrt(2/z),
//    and one integration by parts each for the higher moments:
//      M_1 = [(E(1) - 1)/(2 pi i) + q M_0] / z,   M_2 = [(E(1) - M_0)/(2 pi i) + q M_1] / z.
//  * near tap, z < 1: 8-point Gauss-Legendre on panels spanning at most one phase cycle
//    (half a cycle in FP64).
// Phases with large arguments are reduced modulo 2 in FP64 before sincospi: E(1) =
// exp(i pi (z + 2 (r - k0))) is the same for every tap (q = j - (r - k0) with j integer), and
// q^2/z is formed in FP64 for the near taps.  Everything else runs in the evaluation type T.
//
// k5_interp64, the FP64 evaluation at given points.  GB300 runs FP64 at 1/64 of the FP32 rate (one FP64
// warp instruction takes the SM 16 cycles), so the FP64 instructions are what it costs:
//  * near taps, z >= 1: one table of polynomials (FresnelTable) for d at both ends in place of the series /
//    continued fraction, and the higher moments of all taps from the sums of t, q t, q^2 t, X and q X
//    with t = X conj(sqrt(2z) M_0) (the integrations by parts are linear in M_0);
//  * near taps, z < 1: the sum over the near taps (at most 26) goes inside the integral, which 64
//    Gauss-Legendre nodes then resolve (14 cycles at most): two nodes per lane, Horner over the taps;
//  * far taps: one division-free reciprocal per end and the sums as polynomials in tau^2;
//  * conversions and branch decisions in FP32 and integer arithmetic;
//  * the scalar work (square roots, divisions, the phase at u = 1) lane-parallel: a warp takes a group
//    of points, one per lane, then evaluates them one after another with all lanes on the taps.
// About 65 FP64 instructions per near tap and lane where the form above takes 600.  4096 points, 256 taps,
// |z| <= 84: 1000 -> 270 us, and closer to the exact sums (relative error 3e-15 against 1e-14).  There a step of 32
// taps executes 118 (a warp with near and far taps runs both, and the points' scalar work is in it), and the FP64
// pipe is 87 % busy on an SM that has a block, 69 % over the kernel: 256 blocks at two to an SM leave 48 of 152 SMs
// with one.
// k5_refine keeps the first form for its FP64 step: on a converged candidate whether that step is
// taken hangs on the last bits of P, so another evaluation changes evaluation counts and, along the
// degenerate direction, points.
//
// Refinement (k5_refine), from a seed (r, z), with k0 = floor(r + 1/2) of the seed kept for the
// whole ascent so that P is smooth along the path: up to `steps` FP32 steps, then one FP64 step, of
//   d = H^-1 grad P / P,   H^-1 = (1/(2 pi^2)) [[48, -90], [-90, 180]].
// H is the Hessian of 1 - P/P_peak of an ideal chirp at its peak: an offset (dr, dz) leaves a phase
// error 2 pi (dr u + dz u^2/2) over the observation, and 1 - P/P_peak is to second order its
// variance over u in [0, 1], pi^2 (dr^2/3 + dr dz/3 + 4 dz^2/45).  The step is scaled down to
// |dr| <= 1/4, |dz| <= 1, then halved (at most three times) until P does not decrease; when no
// such step exists the ascent stops.
#include <algorithm>
#include <cmath>

#include "fdas_internal.cuh"
#include "fresnel_table.cuh"
#include "tap_range.cuh"

namespace fdas {

namespace {

constexpr double PI_D = 3.14159265358979323846;
constexpr int WARPS_PER_BLOCK = 4;
constexpr double INV_2PI = 1.0 / (2.0 * PI_D);
constexpr int K5_WARPS = 8;              // warps per block (k5_interp64)
constexpr int K5_GROUP_MAX = 8;          // points per warp (k5_interp64)

struct GL8 {
    double x[8];
    double w[8];
};
struct GL64 {                            // the positive half of the 64 symmetric nodes
    double x[32];
    double w[32];
};

template <typename T>
struct cx {
    T re, im;
};
template <typename T>
__device__ __forceinline__ cx<T> operator+(cx<T> a, cx<T> b) {
    return {a.re + b.re, a.im + b.im};
}
template <typename T>
__device__ __forceinline__ cx<T> operator-(cx<T> a, cx<T> b) {
    return {a.re - b.re, a.im - b.im};
}
template <typename T>
__device__ __forceinline__ cx<T> operator*(cx<T> a, cx<T> b) {
    return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
template <typename T>
__device__ __forceinline__ cx<T> scale(T s, cx<T> a) {
    return {s * a.re, s * a.im};
}
template <typename T>
__device__ __forceinline__ cx<T> conjg(cx<T> a) {
    return {a.re, -a.im};
}
// a * conj(b)
template <typename T>
__device__ __forceinline__ cx<T> mul_conj(cx<T> a, cx<T> b) {
    return {a.re * b.re + a.im * b.im, a.im * b.re - a.re * b.im};
}
// a / (2 pi i) = -i a / (2 pi)
template <typename T>
__device__ __forceinline__ cx<T> over_2pi_i(cx<T> a) {
    const T s = T(1.0 / (2.0 * PI_D));
    return {a.im * s, -a.re * s};
}

// Per-precision choices (series lengths, far-tap threshold, continued-fraction depth, panels).
template <typename T>
struct Arith;
template <>
struct Arith<float> {
    static constexpr float cf_a = 72.f;    // continued-fraction depth floor(cf_a / x^2) + cf_b + 1
    static constexpr int cf_b = 4;
    static constexpr int series_terms = 20;
    static constexpr float far_c = 6.f;
    static constexpr int ibp_terms = 5;
    static constexpr int gl_mult = 1;
    static constexpr float series_max = 1.5f;   // power series for |s| <= series_max
    __device__ static __forceinline__ void scpi(float x, float *s, float *c) { sincospif(x, s, c); }
};
template <>
struct Arith<double> {
    static constexpr double cf_a = 260.0;
    static constexpr int cf_b = 6;
    static constexpr int series_terms = 48;
    static constexpr double far_c = 12.0;
    static constexpr int ibp_terms = 7;
    static constexpr int gl_mult = 2;
    static constexpr double series_max = 2.5;
    __device__ static __forceinline__ void scpi(double x, double *s, double *c) { sincospi(x, s, c); }
};

// exp(i pi x) for an FP64 argument of any size: exact reduction to [-1, 1], then sincospi in T.
template <typename T>
__device__ __forceinline__ cx<T> expipi(double x) {
    const double red = x - 2.0 * rint(0.5 * x);
    T s, c;
    Arith<T>::scpi((T)red, &s, &c);
    return {c, s};
}

// Power-series coefficients of F(s) / s = sum_k x^k / (k! (2k+1)), x = i pi s^2 / 2.
template <int N>
struct SeriesCoef {
    double c[N];
    constexpr SeriesCoef() : c() {
        double f = 1.0;   // k!
        for (int k = 0; k < N; k++) {
            if (k > 0) f *= k;
            c[k] = 1.0 / (f * (2 * k + 1));
        }
    }
};

// F(s) = C(s) + i S(s) as c + d exp(i pi s^2 / 2).
template <typename T>
__device__ void fresnel_end(T s, cx<T> &c, cx<T> &d) {
    const T a = fabs(s);
    if (a <= Arith<T>::series_max) {
        // Horner in the purely imaginary x = i pi s^2/2: S <- S x + c_k
        constexpr int N = Arith<T>::series_terms;
        constexpr SeriesCoef<N> sc;
        const T h = T(PI_D / 2) * s * s;
        cx<T> S = {T(sc.c[N - 1]), T(0)};
#pragma unroll
        for (int k = N - 2; k >= 0; k--) S = {T(sc.c[k]) - S.im * h, S.re * h};
        c = {s * S.re, s * S.im};
        d = {T(0), T(0)};
        return;
    }
    const T sg = s > T(0) ? T(1) : T(-1);
    // K(w) = 1/(w + (1/2)/(w + 1/(w + (3/2)/(w + ...)))), w = (sqrt(pi)/2)(1 - i)|s|, evaluated
    // from a fixed depth upwards (the depth falls as 1/s^2 for a fixed relative accuracy).  The
    // tail t_k = w + a_k / t_{k+1}, a_k = (k-1)/2, is carried as the ratio p/q
    // (p <- w p + a_k q, q <- p), so the only division is the last one.  |p| grows to at most
    // about 1e20 (FP32, |s| just above 1.5) or 1e92 (FP64), inside either format's range.
    const T hw = T(0.88622692545275801365) * a;
    const cx<T> w = {hw, -hw};
    const int depth = (int)(Arith<T>::cf_a / (a * a)) + Arith<T>::cf_b + 1;
    cx<T> p = w, q = {T(1), T(0)};
    for (int k = depth; k >= 2; k--) {
        const T ak = T(0.5) * T(k - 1);
        const cx<T> pn = {w.re * p.re - w.im * p.im + ak * q.re, w.re * p.im + w.im * p.re + ak * q.im};
        q = p;
        p = pn;
    }
    // K = 1 / t_1 = q / p, with both scaled to |p| ~ 1 first so |p|^2 cannot overflow
    const T ps = T(1) / (fabs(p.re) + fabs(p.im));
    p = scale(ps, p);
    q = scale(ps, q);
    const T inv = T(1) / (p.re * p.re + p.im * p.im);
    const cx<T> K = {(q.re * p.re + q.im * p.im) * inv, (q.im * p.re - q.re * p.im) * inv};
    const T nrm = T(0.28209479177387814347);   // 1 / (2 sqrt(pi))
    c = {T(0.5) * sg, T(0.5) * sg};
    d = {-sg * nrm * (K.re - K.im), -sg * nrm * (K.re + K.im)};
}

// What every tap of one evaluation shares (z already folded to z >= 0).
template <typename T>
struct TapCtx {
    double zz;      // |z|
    double dlt;     // q = j - dlt for tap offset j (folded)
    double inv_z;   // 1/zz (zz >= 1)
    T zf;           // zz in T
    T ks;           // sqrt(2/zz)
    T rs2z;         // 1/sqrt(2 zz)
    double dfar;    // far-tap threshold on min |v|
    cx<T> E1;       // E(1) = exp(i pi (zz + 2 dlt)), the same for every tap
};

// Integration-by-parts end term: (m0, m1, m2) at one end u of [0, 1], without the factor E(u).
template <typename T>
__device__ __forceinline__ void ibp_end(T v, T u, T zf, cx<T> &m0, cx<T> &m1, cx<T> &m2) {
    constexpr double c0[7] = {1, 1, 3, 15, 105, 945, 10395};
    constexpr double c1[7] = {1, 3, 15, 105, 945, 10395, 135135};
    constexpr double c2[7] = {1, 6, 45, 420, 4725, 62370, 945945};
    constexpr int n = Arith<T>::ibp_terms;
    const T inv2pi = T(1.0 / (2.0 * PI_D));
    // w = 1/(2 pi i v) = i wi, t = z/(2 pi i v^2) = i tau: both purely imaginary
    const T wi = -inv2pi / v;
    const T tau = -zf * inv2pi / (v * v);
    cx<T> S0 = {T(c0[n - 1]), T(0)}, S1 = {T(c1[n - 1]), T(0)}, S2 = {T(c2[n - 1]), T(0)};
#pragma unroll
    for (int k = n - 2; k >= 0; k--) {   // S = S * (i tau) + c_k
        S0 = {T(c0[k]) - S0.im * tau, S0.re * tau};
        S1 = {T(c1[k]) - S1.im * tau, S1.re * tau};
        S2 = {T(c2[k]) - S2.im * tau, S2.re * tau};
    }
    const cx<T> wS0 = {-wi * S0.im, wi * S0.re};   // w S0
    const T wi2 = wi * wi;                           // -w^2
    const T wi3 = wi2 * wi;                          // w^3 = -i wi^3
    m0 = wS0;
    // u w S0 - w^2 S1 = u w S0 + wi^2 S1
    m1 = {u * wS0.re + wi2 * S1.re, u * wS0.im + wi2 * S1.im};
    // u^2 w S0 - 2 u w^2 S1 + 2 w^3 S2 = u^2 w S0 + 2 u wi^2 S1 - 2 i wi^3 S2
    m2 = {u * u * wS0.re + T(2) * u * wi2 * S1.re + T(2) * wi3 * S2.im,
          u * u * wS0.im + T(2) * u * wi2 * S1.im - T(2) * wi3 * S2.re};
}

template <typename T>
__device__ void tap_moments(const TapCtx<T> &c, int j, const GL8 &gl, cx<T> &M0, cx<T> &M1, cx<T> &M2) {
    const double q = (double)j - c.dlt;
    const T qf = (T)q;
    const double v0 = -q, v1 = c.zz - q;
    const double D = (q >= 0.0 && q <= c.zz) ? 0.0 : fmin(fabs(v0), fabs(v1));
    if (D >= c.dfar) {
        cx<T> a0, a1, a2, b0, b1, b2;
        ibp_end<T>((T)v1, T(1), c.zf, a0, a1, a2);
        ibp_end<T>((T)v0, T(0), c.zf, b0, b1, b2);
        M0 = c.E1 * a0 - b0;
        M1 = c.E1 * a1 - b1;
        M2 = c.E1 * a2 - b2;
        return;
    }
    if (c.zz >= 1.0) {
        const T s0 = -qf * c.ks;
        const T s1 = (c.zf - qf) * c.ks;
        cx<T> c0, d0, c1, d1;
        fresnel_end<T>(s0, c0, d0);
        fresnel_end<T>(s1, c1, d1);
        const cx<T> ph = expipi<T>(-q * q * c.inv_z);
        M0 = scale(c.rs2z, (c1 - c0) * ph + d1 * c.E1 - d0);
        const T iz = (T)c.inv_z;
        const cx<T> one = {T(1), T(0)};
        M1 = scale(iz, over_2pi_i(c.E1 - one) + scale(qf, M0));
        M2 = scale(iz, over_2pi_i(c.E1 - M0) + scale(qf, M1));
        return;
    }
    // |z| < 1, |q| < dfar + 1: panels of at most one (FP64: half a) phase cycle
    const int panels = max(1, (int)ceil(fabs(q) + c.zz)) * Arith<T>::gl_mult;
    const T h = T(1) / T(panels);
    cx<T> a0 = {T(0), T(0)}, a1 = a0, a2 = a0;
    for (int p = 0; p < panels; p++) {
        const T mid = (T(p) + T(0.5)) * h;
#pragma unroll
        for (int g = 0; g < 8; g++) {
            const T u = mid + T(0.5) * h * (T)gl.x[g];
            T s, co;
            Arith<T>::scpi(u * (c.zf * u - T(2) * qf), &s, &co);
            const T wt = T(0.5) * h * (T)gl.w[g];
            const cx<T> e = {wt * co, wt * s};
            a0 = a0 + e;
            a1 = a1 + scale(u, e);
            a2 = a2 + scale(u * u, e);
        }
    }
    M0 = a0;
    M1 = a1;
    M2 = a2;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Points the evaluation accepts (anything else gives NaN): finite, |r| < 2^52, |z| < 2^20 and the
// window no further than 2^24 bins from r.
__device__ __forceinline__ bool point_ok(double r, double z, int64_t k0) {
    return isfinite(r) && isfinite(z) && fabs(r) < 4.5e15 && fabs(z) < 1048576.0 &&
           fabs(r - (double)k0) < 16777216.0;
}

// P, dP/dr, dP/dz at (r, z) with the window anchored at k0 (warp-collective; every lane returns
// the same values).
template <typename T>
__device__ void eval_point(const float2 *__restrict__ xhat, int64_t nb, int m, int64_t k0, double r, double z,
                           const GL8 &gl, T &P, T &dPdr, T &dPdz) {
    const int lane = threadIdx.x & 31;
    const bool neg = z < 0.0;
    TapCtx<T> c;
    c.zz = fabs(z);
    const double dlt = r - (double)k0;
    c.dlt = neg ? -dlt : dlt;
    c.zf = (T)c.zz;
    const bool big = c.zz >= 1.0;
    c.inv_z = big ? 1.0 / c.zz : 0.0;
    c.ks = big ? (T)sqrt(2.0 / c.zz) : T(0);
    c.rs2z = big ? (T)(1.0 / sqrt(2.0 * c.zz)) : T(0);
    c.dfar = (double)Arith<T>::far_c * fmax(1.0, sqrt(c.zz));
    c.E1 = expipi<T>(c.zz + 2.0 * c.dlt);
    cx<T> A = {T(0), T(0)}, Y1 = A, Y2 = A;
    for (int t = lane; t < m; t += 32) {
        const int j = t - m / 2;
        const int64_t k = k0 + j;
        if (k < 0 || k >= nb) continue;
        const float2 xv = __ldg(xhat + k);
        const cx<T> X = {(T)xv.x, (T)xv.y};
        cx<T> M0, M1, M2;
        tap_moments<T>(c, neg ? -j : j, gl, M0, M1, M2);
        if (neg) {
            M0 = conjg(M0);
            M1 = conjg(M1);
            M2 = conjg(M2);
        }
        A = A + mul_conj(X, M0);
        Y1 = Y1 + mul_conj(X, M1);
        Y2 = Y2 + mul_conj(X, M2);
    }
    A.re = warp_sum(A.re);
    A.im = warp_sum(A.im);
    Y1.re = warp_sum(Y1.re);
    Y1.im = warp_sum(Y1.im);
    Y2.re = warp_sum(Y2.re);
    Y2.im = warp_sum(Y2.im);
    // dA/dr = sum X conj(2 pi i M_1) = -2 pi i Y1,  dA/dz = sum X conj(i pi M_2) = -i pi Y2
    const T tp = T(2.0 * PI_D), pi = T(PI_D);
    const cx<T> Ar = {tp * Y1.im, -tp * Y1.re};
    const cx<T> Az = {pi * Y2.im, -pi * Y2.re};
    P = A.re * A.re + A.im * A.im;
    dPdr = T(2) * (A.re * Ar.re + A.im * Ar.im);
    dPdz = T(2) * (A.re * Az.re + A.im * Az.im);
}

template <typename T>
__global__ void __launch_bounds__(32 * WARPS_PER_BLOCK)
    k5_interp(const float2 *__restrict__ xhat, int64_t nb, int m, const fdas_cand *__restrict__ pts,
              const int64_t *__restrict__ k0s, int n, double *__restrict__ out, GL8 gl) {
    const int i = (int)((blockIdx.x * (unsigned)blockDim.x + threadIdx.x) >> 5);
    if (i >= n) return;
    const double r = pts[i].r, z = pts[i].z;
    const int64_t k0 = k0s ? k0s[i] : (isfinite(r) && fabs(r) < 4.5e15 ? (int64_t)floor(r + 0.5) : 0);
    T P = T(NAN), gr = T(NAN), gz = T(NAN);
    if (point_ok(r, z, k0)) eval_point<T>(xhat, nb, m, k0, r, z, gl, P, gr, gz);
    if ((threadIdx.x & 31) == 0) {
        out[3 * (size_t)i + 0] = (double)P;
        out[3 * (size_t)i + 1] = (double)gr;
        out[3 * (size_t)i + 2] = (double)gz;
    }
}

// ---------------------------------------------------------------------------------------
// FP64 evaluation

constexpr float FAR_C64 = 12.f;

template <typename V>
__device__ __forceinline__ V from_lane(V v, int l) {
    return __shfl_sync(0xffffffffu, v, l);
}

struct Setup64 {
    int64_t k0;
    double zz, dlt;     // |z|; q = j - dlt for tap offset j (folded)
    double inv_z, inv_z_lo;   // 1/zz as a pair (zz >= 1)
    double ks;          // sqrt(2/zz)
    cx<double> E1;      // E(1)
    int neg;
};

// exp(i pi x), x reduced to [-1, 1] modulo 2 (exact) first
__device__ __forceinline__ double mod2(double x) { return x - 2.0 * rint(0.5 * x); }
__device__ __forceinline__ cx<double> expipi64(double x) {
    double s, c;
    sincospi(mod2(x), &s, &c);
    return {c, s};
}

__device__ __forceinline__ void setup64(Setup64 &c, int64_t k0, double r, double z) {
    c.neg = z < 0.0;
    c.k0 = k0;
    c.zz = fabs(z);
    const double dlt = r - (double)k0;
    c.dlt = c.neg ? -dlt : dlt;
    const bool big = c.zz >= 1.0;
    c.inv_z = big ? 1.0 / c.zz : 0.0;
    c.inv_z_lo = fma(-c.zz, c.inv_z, 1.0) * c.inv_z;
    c.ks = big ? sqrt(2.0 / c.zz) : 0.0;
    c.E1 = expipi64(c.zz + 2.0 * c.dlt);
}
__device__ __forceinline__ Setup64 from_lane(const Setup64 &s, int l) {
    Setup64 c;
    c.k0 = from_lane((long long)s.k0, l);
    c.zz = from_lane(s.zz, l);
    c.dlt = from_lane(s.dlt, l);
    c.inv_z = from_lane(s.inv_z, l);
    c.inv_z_lo = from_lane(s.inv_z_lo, l);
    c.ks = from_lane(s.ks, l);
    c.E1.re = from_lane(s.E1.re, l);
    c.E1.im = from_lane(s.E1.im, l);
    c.neg = from_lane(s.neg, l);
    return c;
}

// A float widened to FP64 with integer operations (positive or negative normal values): FP64
// conversions run at the FP64 rate.
__device__ __forceinline__ double widen(float f) {
    const unsigned b = __float_as_uint(f);
    const unsigned hi = (b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u);
    return __hiloint2double((int)hi, (int)(b << 29));
}
// any float (zeros, subnormals, infinities and NaN converted)
__device__ __forceinline__ double widen_any(float f) {
    const unsigned e = __float_as_uint(f) & 0x7f800000u;
    return e == 0u || e == 0x7f800000u ? (double)f : widen(f);
}

// -sgn(s) G(|s|) from the table (shared memory, [coefficient][interval]); sf: s to FP32 accuracy.
__device__ __forceinline__ cx<double> fresnel_d(const double2 *tab, double s, float sf) {
    const FresnelSpot at = fresnel_spot(fabsf(sf));
    const double u = fabs(s) - widen(at.centre);
    const double2 *p = tab + at.idx;
    double2 c = p[(FRESNEL_TERMS - 1) * FRESNEL_INTERVALS];
    double re = c.x, im = c.y;
#pragma unroll
    for (int k = FRESNEL_TERMS - 2; k >= 0; k--) {
        c = p[k * FRESNEL_INTERVALS];
        re = fma(re, u, c.x);
        im = fma(im, u, c.y);
    }
    // the sign by integer operations on the high words
    const int flip = (~__double2hiint(s)) & 0x80000000;
    return {__hiloint2double(__double2hiint(re) ^ flip, __double2loint(re)),
            __hiloint2double(__double2hiint(im) ^ flip, __double2loint(im))};
}

// Integration-by-parts end term at u = U (0 or 1), without E(u): the sums of ibp_end with 7 (S1, S2)
// and 8 (S0) terms, real and imaginary parts as polynomials in tau^2.  vf: v in FP32.
template <int U>
__device__ __forceinline__ void ibp_end64(double v, float vf, double zz, cx<double> &m0, cx<double> &m1, cx<double> &m2) {
    // 1/v: an FP32 seed (relative error e below 2^-20), then r (1 + e + e^2) (Newton's iteration, third order)
    double r = widen(__frcp_rn(vf));
    const double e = fma(-v, r, 1.0);
    r = fma(r, fma(e, e, e), r);
    const double wi = -INV_2PI * r;
    const double tau = zz * (wi * r);
    const double t2 = tau * tau;
    const double s1r = fma(t2, fma(t2, fma(t2, -135135.0, 945.0), -15.0), 1.0);
    const double s1i = tau * fma(t2, fma(t2, 10395.0, -105.0), 3.0);
    const double s2r = fma(t2, fma(t2, fma(t2, -945945.0, 4725.0), -45.0), 1.0);
    const double s2i = tau * fma(t2, fma(t2, 62370.0, -420.0), 6.0);
    const double s0r = fma(-tau, s1i, 1.0), s0i = tau * s1r;
    const double wi2 = wi * wi, wi3 = 2.0 * wi2 * wi;
    m0 = {-wi * s0i, wi * s0r};
    if (U == 1) {
        m1 = {fma(wi2, s1r, m0.re), fma(wi2, s1i, m0.im)};
        m2 = {fma(wi3, s2i, fma(wi2, s1r, m1.re)), fma(-wi3, s2r, fma(wi2, s1i, m1.im))};
    } else {
        m1 = {wi2 * s1r, wi2 * s1i};
        m2 = {wi3 * s2i, -wi3 * s2r};
    }
}

// acc += a conj(b)
__device__ __forceinline__ void mac_conj(cx<double> &acc, cx<double> a, cx<double> b) {
    acc.re = fma(a.re, b.re, fma(a.im, b.im, acc.re));
    acc.im = fma(a.im, b.re, fma(-a.re, b.im, acc.im));
}
// E a - b
__device__ __forceinline__ cx<double> mul_sub(cx<double> E, cx<double> a, cx<double> b) {
    return {fma(E.re, a.re, fma(-E.im, a.im, -b.re)), fma(E.re, a.im, fma(E.im, a.re, -b.im))};
}

// P and its gradient from the three sums: dA/dr = sum X conj(2 pi i M_1) = -2 pi i Y1,
// dA/dz = sum X conj(i pi M_2) = -i pi Y2
struct Value64 {
    double P, dPdr, dPdz;
};
__device__ __forceinline__ Value64 value_of(cx<double> A, cx<double> Y1, cx<double> Y2) {
    const cx<double> Ar = {2.0 * PI_D * Y1.im, -2.0 * PI_D * Y1.re};
    const cx<double> Az = {PI_D * Y2.im, -PI_D * Y2.re};
    return {A.re * A.re + A.im * A.im, 2.0 * (A.re * Ar.re + A.im * Ar.im), 2.0 * (A.re * Az.re + A.im * Az.im)};
}

// The value at one point in FP64 (warp-collective; every lane returns the same values).  z < 0 is
// folded by conjugation: sum X conj(M(q, z)) = conj(sum conj(X) conj(M(-q, -z))).
// Near taps with z >= 1: with t = X conj(sqrt(2z) M_0), the higher moments of all of them follow
// from sum t, sum q t, sum q^2 t, sum X and sum q X (the two integrations by parts are linear in M_0).
__device__ Value64 eval64(const float2 *__restrict__ xhat, int64_t nb, int m, const Setup64 &c,
                                const double2 *tab, const GL64 &gl) {
    const int lane = threadIdx.x & 31;
    const cx<double> zero = {0.0, 0.0};
    cx<double> A = zero, Y1 = zero, Y2 = zero;                             // far taps (and the z < 1 integral)
    const float zf = (float)c.zz, ksf = (float)c.ks;
    const int di = (int)rint(c.dlt);                                       // q = (j - di) - df in FP32
    const float df = (float)(c.dlt - (double)di);
    const bool big = c.zz >= 1.0;
    const float dfar = FAR_C64 * fmaxf(1.f, sqrtf(zf));
    const int half = m / 2;
    const TapRange on = taps_on_spectrum(c.k0, m, nb);                     // unfolded offsets
    cx<double> T0 = zero, T1 = zero, T2 = zero, SX = zero, SqX = zero;     // near taps, z >= 1
    int jl = 1, jh = 0;                                                    // near taps, z < 1
    if (!big) {
        jl = di + (int)ceilf(df - dfar);
        jh = di + (int)floorf(df + zf + dfar);
    }
    for (int t = lane; t < m; t += 32) {
        const int ju = t - half;
        if (ju < on.lo || ju > on.hi) continue;
        const int j = c.neg ? -ju : ju;
        if (j >= jl && j <= jh) continue;
        const float2 xv = __ldg(xhat + c.k0 + ju);
        const cx<double> X = {widen_any(xv.x), c.neg ? -widen_any(xv.y) : widen_any(xv.y)};
        const double q = widen_any((float)j) - c.dlt;
        const float qf = (float)(j - di) - df;
        if (!big || fmaxf(-qf, qf - zf) >= dfar) {
            cx<double> a0, a1, a2, b0, b1, b2;
            ibp_end64<1>(c.zz - q, zf - qf, c.zz, a0, a1, a2);
            ibp_end64<0>(-q, -qf, c.zz, b0, b1, b2);
            mac_conj(A, X, mul_sub(c.E1, a0, b0));
            mac_conj(Y1, X, mul_sub(c.E1, a1, b1));
            mac_conj(Y2, X, mul_sub(c.E1, a2, b2));
        } else {
            const double s0 = -q * c.ks, s1 = (c.zz - q) * c.ks;
            const cx<double> d0 = fresnel_d(tab, s0, qf * ksf);
            const cx<double> d1 = fresnel_d(tab, s1, (zf - qf) * ksf);
            cx<double> M = mul_sub(c.E1, d1, d0);
            if ((__double2hiint(s0) < 0) != (__double2hiint(s1) < 0)) {    // 0 < q <= z: c1 - c0 = 1 + i
                // q^2/z with its rounding errors carried, then modulo 2
                const double p = q * q, pl = fma(q, q, -p);
                const double y = p * c.inv_z;
                const double yl = fma(p, c.inv_z, -y) + fma(p, c.inv_z_lo, pl * c.inv_z);
                double si, co;
                sincospi(-(mod2(y) + yl), &si, &co);
                M.re += co - si;
                M.im += co + si;
            }
            const cx<double> tt = {fma(X.re, M.re, X.im * M.im), fma(X.im, M.re, -X.re * M.im)};
            const double q2 = q * q;
            T0 = T0 + tt;
            T1 = {fma(q, tt.re, T1.re), fma(q, tt.im, T1.im)};
            T2 = {fma(q2, tt.re, T2.re), fma(q2, tt.im, T2.im)};
            SX = SX + X;
            SqX = {fma(q, X.re, SqX.re), fma(q, X.im, SqX.im)};
        }
    }
    if (big) {
        // M_1 = K1 + (q/z) M_0, K1 = (E1 - 1)/(2 pi i z);  M_2 = E1/(2 pi i z) - M_0/(2 pi i z) + (q/z) M_1
        const double iz = c.inv_z, rs = 0.5 * c.ks;                        // 1/sqrt(2z) = sqrt(2/z)/2
        const cx<double> K1 = scale(iz, over_2pi_i(c.E1 - cx<double>{1.0, 0.0})), K2 = scale(iz, over_2pi_i(c.E1));
        T0 = scale(rs, T0);
        T1 = scale(rs * iz, T1);
        T2 = scale(rs * iz * iz, T2);
        A = A + T0;
        mac_conj(Y1, SX, K1);
        Y1 = Y1 + T1;
        mac_conj(Y2, SX, K2);
        mac_conj(Y2, scale(iz, SqX), K1);
        // - conj(1/(2 pi i z)) T0 = -(i iz / (2 pi)) T0
        Y2 = Y2 + T2 + cx<double>{iz * INV_2PI * T0.im, -iz * INV_2PI * T0.re};
    } else {
        // int_0^1 u^p exp(-i pi z u^2) sum_j X_j exp(2 pi i (j - dlt) u) du: lane l holds nodes +-x[l];
        // Horner over j from jh down to jl in exp(2 pi i u)
        const TapRange near = taps_between(on, c.neg, jl, jh);
        const int jlo = near.lo, jhi = near.hi;
        const double xg = gl.x[lane], wg = 0.5 * gl.w[lane];
        const double u0 = 0.5 * (1.0 - xg), u1 = 0.5 * (1.0 + xg);
        const cx<double> w0 = expipi64(2.0 * u0), w1 = expipi64(2.0 * u1);
        cx<double> B0 = zero, B1 = zero;
        for (int j = jhi; j >= jlo; j--) {
            const float2 xv = __ldg(xhat + c.k0 + (c.neg ? -j : j));
            const cx<double> X = {widen_any(xv.x), c.neg ? -widen_any(xv.y) : widen_any(xv.y)};
            B0 = {fma(B0.re, w0.re, fma(-B0.im, w0.im, X.re)), fma(B0.re, w0.im, fma(B0.im, w0.re, X.im))};
            B1 = {fma(B1.re, w1.re, fma(-B1.im, w1.im, X.re)), fma(B1.re, w1.im, fma(B1.im, w1.re, X.im))};
        }
        if (jlo <= jhi) {
            const double off = 2.0 * ((double)jlo - c.dlt);
            const cx<double> e0 = scale(wg, expipi64(u0 * (off - c.zz * u0)) * B0);
            const cx<double> e1 = scale(wg, expipi64(u1 * (off - c.zz * u1)) * B1);
            A = A + e0 + e1;
            Y1 = Y1 + scale(u0, e0) + scale(u1, e1);
            Y2 = Y2 + scale(u0 * u0, e0) + scale(u1 * u1, e1);
        }
    }
    A.re = warp_sum(A.re);
    A.im = warp_sum(A.im);
    Y1.re = warp_sum(Y1.re);
    Y1.im = warp_sum(Y1.im);
    Y2.re = warp_sum(Y2.re);
    Y2.im = warp_sum(Y2.im);
    if (c.neg) {
        A.im = -A.im;
        Y1.im = -Y1.im;
        Y2.im = -Y2.im;
    }
    return value_of(A, Y1, Y2);
}

// One evaluation for every lane of the warp with `on` set, at (r, z) anchored at k0.
__device__ __forceinline__ void eval64_lanes(const float2 *__restrict__ xhat, int64_t nb, int m, bool on, int64_t k0, double r,
                                             double z, const double2 *tab, const GL64 &gl, Value64 &v) {
    Setup64 mine{};
    if (on) setup64(mine, k0, r, z);
    for (unsigned todo = __ballot_sync(0xffffffffu, on); todo; todo &= todo - 1) {
        const int l = __ffs(todo) - 1;
        const Value64 got = eval64(xhat, nb, m, from_lane(mine, l), tab, gl);
        if ((int)(threadIdx.x & 31) == l) v = got;
    }
}

__device__ __forceinline__ void load_table(double2 *tab) {
    for (int i = threadIdx.x; i < FRESNEL_TERMS * FRESNEL_INTERVALS; i += blockDim.x)
        tab[i] = reinterpret_cast<const double2 *>(fresnel_table.c)[i];
    __syncthreads();
}

__device__ __forceinline__ int64_t anchor_of(double r) {
    return isfinite(r) && fabs(r) < 4.5e15 ? (int64_t)floor(r + 0.5) : 0;
}

// Interpolated power in FP64, `group` consecutive points per warp.
__global__ void __launch_bounds__(32 * K5_WARPS, 2)
    k5_interp64(const float2 *__restrict__ xhat, int64_t nb, int m, const fdas_cand *__restrict__ pts,
                const int64_t *__restrict__ k0s, int n, int group, double *__restrict__ out, GL64 gl) {
    extern __shared__ double2 tab[];
    load_table(tab);
    const int lane = threadIdx.x & 31;
    const int64_t i = ((int64_t)blockIdx.x * K5_WARPS + (threadIdx.x >> 5)) * group + lane;
    const bool mine = lane < group && i < n;
    const double r = mine ? pts[i].r : NAN, z = mine ? pts[i].z : NAN;
    const int64_t k0 = mine && k0s ? k0s[i] : anchor_of(r);
    Value64 v = {NAN, NAN, NAN};
    eval64_lanes(xhat, nb, m, point_ok(r, z, k0), k0, r, z, tab, gl, v);
    if (mine) {
        out[3 * (size_t)i + 0] = v.P;
        out[3 * (size_t)i + 1] = v.dPdr;
        out[3 * (size_t)i + 2] = v.dPdz;
    }
}

// The preconditioned step (see the header comment); false when there is none.
__device__ __forceinline__ bool ascent_step(double P, double gr, double gz, double &dr, double &dz) {
    if (!(P > 0.0)) return false;
    const double s = 1.0 / (2.0 * PI_D * PI_D * P);
    dr = (48.0 * gr - 90.0 * gz) * s;
    dz = (-90.0 * gr + 180.0 * gz) * s;
    const double sc = fmax(fmax(4.0 * fabs(dr), fabs(dz)), 1.0);
    dr /= sc;
    dz /= sc;
    return isfinite(dr) && isfinite(dz);
}

constexpr int HALVINGS = 4;   // tries per step: d, d/2, d/4, d/8

__global__ void __launch_bounds__(32 * WARPS_PER_BLOCK)
    k5_refine(const float2 *__restrict__ xhat, int64_t nb, int m, const fdas_cand *__restrict__ in, int n,
              int steps, fdas_cand *__restrict__ out, double *__restrict__ pw, int32_t *__restrict__ evals_out,
              GL8 gl) {
    const int c = (int)((blockIdx.x * (unsigned)blockDim.x + threadIdx.x) >> 5);
    if (c >= n) return;
    double r = in[c].r, z = in[c].z;
    const int64_t k0 = (isfinite(r) && fabs(r) < 4.5e15) ? (int64_t)floor(r + 0.5) : 0;
    int evals = 0;
    double Pd = NAN, grd = NAN, gzd = NAN;
    if (point_ok(r, z, k0)) {
        float P, gr, gz;
        eval_point<float>(xhat, nb, m, k0, r, z, gl, P, gr, gz);
        evals++;
        for (int s = 0; s < steps; s++) {
            double dr, dz;
            if (!ascent_step(P, gr, gz, dr, dz)) break;
            bool ok = false;
            float P2, gr2, gz2;
            for (int h = 0; h < HALVINGS; h++) {
                eval_point<float>(xhat, nb, m, k0, r + dr, z + dz, gl, P2, gr2, gz2);
                evals++;
                if (P2 >= P) {
                    ok = true;
                    break;
                }
                dr *= 0.5;
                dz *= 0.5;
            }
            if (!ok) break;
            r += dr;
            z += dz;
            P = P2;
            gr = gr2;
            gz = gz2;
        }
        // the final step in FP64
        eval_point<double>(xhat, nb, m, k0, r, z, gl, Pd, grd, gzd);
        evals++;
        double dr, dz;
        if (ascent_step(Pd, grd, gzd, dr, dz)) {
            for (int h = 0; h < HALVINGS; h++) {
                double P2, gr2, gz2;
                eval_point<double>(xhat, nb, m, k0, r + dr, z + dz, gl, P2, gr2, gz2);
                evals++;
                if (P2 >= Pd) {
                    r += dr;
                    z += dz;
                    Pd = P2;
                    grd = gr2;
                    gzd = gz2;
                    break;
                }
                dr *= 0.5;
                dz *= 0.5;
            }
        }
    }
    if ((threadIdx.x & 31) == 0) {
        out[c].r = r;
        out[c].z = z;
        if (pw) {
            pw[3 * (size_t)c + 0] = Pd;
            pw[3 * (size_t)c + 1] = grd;
            pw[3 * (size_t)c + 2] = gzd;
        }
        if (evals_out) evals_out[c] = evals;
    }
}

GL8 gl8() {
    static GL8 g = [] {
        GL8 t;
        gauss_legendre(8, t.x, t.w);
        return t;
    }();
    return g;
}

unsigned blocks_for(int n) { return (unsigned)((n + WARPS_PER_BLOCK - 1) / WARPS_PER_BLOCK); }

const GL64 &gl64() {
    static const GL64 g = [] {
        double x[64], w[64];
        gauss_legendre(64, x, w);
        GL64 t;
        for (int i = 0; i < 32; i++) {
            t.x[i] = x[i];
            t.w[i] = w[i];
        }
        return t;
    }();
    return g;
}

// Points per warp: as many as leave about 12 warps per SM busy (a group shares the scalar FP64 work).
int group_size(const Plan &p, int n) {
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p.device >= 0 ? p.device : 0);
    return std::max(1, std::min(K5_GROUP_MAX, n / (12 * std::max(sms, 1))));
}
constexpr size_t TABLE_BYTES = sizeof(double2) * FRESNEL_TERMS * FRESNEL_INTERVALS;
static_assert(TABLE_BYTES <= 48 * 1024, "the table fits the default shared-memory limit");


}  // namespace

cudaError_t launch_interp(Plan &p, const float2 *d_x, const fdas_cand *d_pts, const int64_t *d_k0, int n, bool fp64,
                          double *d_out, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    if (fp64) {
        const int g = group_size(p, n);
        const unsigned blocks = (unsigned)((n + (int64_t)K5_WARPS * g - 1) / (K5_WARPS * g));
        k5_interp64<<<blocks, 32 * K5_WARPS, TABLE_BYTES, st>>>(d_x, p.nb, p.m, d_pts, d_k0, n, g, d_out, gl64());
    } else {
        k5_interp<float><<<blocks_for(n), 32 * WARPS_PER_BLOCK, 0, st>>>(d_x, p.nb, p.m, d_pts, d_k0, n, d_out, gl8());
    }
    p.prof.launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_refine(Plan &p, const float2 *d_x, const fdas_cand *d_in, int n, int steps, fdas_cand *d_out,
                          double *d_power, int32_t *d_evals, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k5_refine<<<blocks_for(n), 32 * WARPS_PER_BLOCK, 0, st>>>(d_x, p.nb, p.m, d_in, n, steps, d_out, d_power,
                                                              d_evals, gl8());
    p.prof.launches += 1;
    return cudaGetLastError();
}

}  // namespace fdas
