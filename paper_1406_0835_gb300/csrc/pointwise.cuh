// Pointwise finite-T functional math, shared by host (checks) and device.
//
//   tfunc_eval   xi, zeta, A, B of t and their t-derivatives from the table
//   enhance      F(x) and dF/dx of the enhancement factors (Sec. III B)
//   fs_point     f_s, df_s/dn and W = df_s/d(grad n) / grad n at one point
//                (Eqs. (fTF), (vTF), (FGGA), (s_s), (s_0defn), (vftGGA))
//   pz81_point   Perdew-Zunger LDA eps_xc and v_xc (Sec. IV, Eq. (vxc1) at T = 0)
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#include "ffmath.cuh"
#include "ofdft_internal.h"

namespace ofdft {

#ifdef __CUDACC__
#define OF_HD __host__ __device__ __forceinline__
#else
#define OF_HD inline
#endif

// t = m 2^e with m in [1, 2); returns m and 2^-e.
OF_HD double split_pow2(double t, int &e, double &inv2e)
{
    int64_t b;
#ifdef __CUDA_ARCH__
    b = __double_as_longlong(t);
#else
    memcpy(&b, &t, 8);
#endif
    e = (int)((b >> 52) & 0x7ff) - 1023;
    int64_t mb = (b & 0x000fffffffffffffLL) | 0x3ff0000000000000LL;
    int64_t ib = (int64_t)(1023 - e) << 52;
    double m;
#ifdef __CUDA_ARCH__
    m = __longlong_as_double(mb);
    inv2e = __longlong_as_double(ib);
#else
    memcpy(&m, &mb, 8);
    memcpy(&inv2e, &ib, 8);
#endif
    return m;
}

OF_HD float split_pow2(float t, int &e, float &inv2e)
{
    int32_t b;
#ifdef __CUDA_ARCH__
    b = __float_as_int(t);
#else
    memcpy(&b, &t, 4);
#endif
    e = (int)((b >> 23) & 0xff) - 127;
    int32_t mb = (b & 0x007fffff) | 0x3f800000;
    int32_t ib = (int32_t)(127 - e) << 23;
    float m;
#ifdef __CUDA_ARCH__
    m = __int_as_float(mb);
    inv2e = __int_as_float(ib);
#else
    memcpy(&m, &mb, 4);
    memcpy(&inv2e, &ib, 4);
#endif
    return m;
}

// n^{-1/3} for n > 0: seed from the exponent split n = m 2^(3q + r), m 2^r in
// [1, 8), with a single-precision power of that factor, then Newton steps
// y <- y (4 - n y^3)/3 (quadratic convergence; 2 steps reach double rounding
// from a ~1e-7 seed, 1 step reaches float rounding).
OF_HD double inv_cbrt(double n)
{
    int e;
    double s;
    double m = split_pow2(n, e, s);
    int q = (e >= 0) ? e / 3 : -((2 - e) / 3);      // floor(e / 3)
    int r = e - 3 * q;                                 // 0, 1, 2
    double mm = m * (double)(1 << r);
    double y = (double)powf((float)mm, -1.0f / 3.0f);
    int64_t ib = (int64_t)(1023 - q) << 52;            // 2^-q
    double sc;
#ifdef __CUDA_ARCH__
    sc = __longlong_as_double(ib);
#else
    memcpy(&sc, &ib, 8);
#endif
    y *= sc;
    for (int k = 0; k < 2; ++k) y = y * (4.0 - n * (y * y * y)) * (1.0 / 3.0);
    return y;
}

OF_HD float inv_cbrt(float n)
{
    float y = powf(n, -1.0f / 3.0f);
    return y * (4.0f - n * (y * y * y)) * (1.0f / 3.0f);
}

// out[0..3] = xi, zeta, A, B; out[4..7] = d/dt of each (nf functions: 2 or 4).
template <typename T, int NF = kTfFuncs>
OF_HD void tfunc_eval(const T *__restrict__ tab, T t, T out[8])
{
    const T pi2 = T(9.8696044010893586188);
    if (!(t >= T(9.5367431640625e-07))) {            // t < 2^-20: Sommerfeld limit
        T t2 = t * t;
        out[0] = T(1) + T(5.0 / 12.0) * pi2 * t2;     // xi = 1 + (5 pi^2/12) t^2
        out[1] = T(5.0 / 6.0) * pi2 * t2;             // zeta = (5 pi^2/6) t^2
        out[2] = T(1) - T(0.75) * pi2 * t2;           // A = 1 - (3 pi^2/4) t^2
        out[3] = T(0.8);                              // B -> 4/5
        out[4] = T(5.0 / 6.0) * pi2 * t;
        out[5] = T(5.0 / 3.0) * pi2 * t;
        out[6] = T(-1.5) * pi2 * t;
        out[7] = T(0);
        return;
    }
    if (t >= T(17179869184.0)) {                      // t >= 2^34: classical gas
        // e^eta = (4/(3 sqrt(pi))) t^{-3/2}; xi = (5/2) t; zeta = (5/3) t (5/2 - eta); h~ = 3
        T eta = T(-0.28468287047291918) - T(1.5) * log(t);
        out[0] = T(2.5) * t;
        out[1] = T(5.0 / 3.0) * t * (T(2.5) - eta);
        out[2] = T(1.2) / t;
        out[3] = T(0);
        out[4] = T(2.5);
        out[5] = T(5.0 / 3.0) * (T(2.5) - eta) + T(2.5);
        out[6] = T(-1.2) / (t * t);
        out[7] = T(0);
        return;
    }
    int e;
    T inv2e;
    T m = split_pow2(t, e, inv2e);
    int sub = (int)((m - T(1)) * T(4));
    T u = T(8) * (m - T(1)) - T(2 * sub + 1);
    const T *c = tab + ((size_t)((e - kTfEmin) * kTfSub + sub) * kTfFuncs) * kTfNc;
    T dudt = T(8) * inv2e;
#pragma unroll
    for (int q = 0; q < NF; ++q) {
        const T *cq = c + q * kTfNc;
        T p = cq[kTfDeg], dp = T(0);
#pragma unroll
        for (int j = kTfDeg - 1; j >= 0; --j) {
            dp = dp * u + p;
            p = p * u + cq[j];
        }
        out[q] = p;
        out[4 + q] = dp * dudt;
    }
}

// Enhancement factor F(x), x = s^2, and dF/dx.
template <typename T>
OF_HD void enhance(const FuncParams &fp, T x, T &F, T &dF)
{
    if (fp.kind == 1) {                       // SGA form, Eq. (SGA-F)
        F = T(1) + T(fp.p0) * x;
        dF = T(fp.p0);
    } else if (fp.kind == 3) {                // KST2 form, Eq. (KST2F)
        T den = T(1) / (T(1) + T(fp.p1) * x);
        F = T(1) + T(fp.p0) * x * den;
        dF = T(fp.p0) * den * den;
    } else {                                  // VT84F, Eq. (VT84F), m = 8, n = 4
        const T mu = T(2.778), al = T(1.2965);
        const T tiny = sizeof(T) == 8 ? T(1e-100) : T(1e-15);
        if (x <= tiny) {                      // removable 0/0 at x = 0
            F = T(1);
            dF = -mu + al + T(5.0 / 3.0);
            return;
        }
        T e1 = exp(-al * x);
        T x2 = x * x;
        T em = -expm1(-al * x2);              // 1 - exp(-al x^2)
        T q = T(1) + mu * x;
        T inv = T(1) / (x * q);               // one division for 1/x and 1/(1 + mu x)
        T rx = q * inv;
        T den = x * inv;
        F = T(1) - mu * x * e1 * den + em * (rx - T(1)) + T(5.0 / 3.0) * x;
        dF = -mu * e1 * (T(1) - al * x - al * mu * x2) * den * den
             + T(2) * al * (T(1) - em) * (T(1) - x) - em * rx * rx + T(5.0 / 3.0);
    }
}

// Output of the non-interacting functional at one point.
template <typename T> struct FsOut {
    T f;      // f_s
    T ts;     // tau0 zeta F_sigma (entropic density T s)
    T dfdn;   // partial f / partial n (without the divergence term)
    T wc;     // W = wc * grad n
    T y13;    // n^{-1/3} (reused by the XC term)
};

// Constants: C_TF = (3/10)(3 pi^2)^{2/3}; (3 pi^2)^{2/3}; cs = 1/(4 (3 pi^2)^{2/3}).
#define OF_K23 9.5707800006273045              /* (3 pi^2)^{2/3} */
#define OF_CTF (0.3 * OF_K23)                      /* (3/10)(3 pi^2)^{2/3}, Eq. (tauTFdefn) */
#define OF_CS (1.0 / (4.0 * OF_K23))               /* s^2 = |grad n|^2 OF_CS / n^{8/3} */

template <typename T>
OF_HD FsOut<T> fs_point(const FuncParams &fp, const T *__restrict__ tab, T temp, T n, T g2)
{
    FsOut<T> o;
    T y = inv_cbrt(n);                                  // n^{-1/3}
    o.y13 = y;
    T y2 = y * y;
    T c13 = n * y2;                                     // n^{1/3}
    T n23 = c13 * c13;
    T rn = y2 * y;                                      // 1/n
    T tau0 = T(OF_CTF) * n * n23;                       // Eq. (tauTFdefn)
    T dtau0 = T(5.0 / 3.0 * OF_CTF) * n23;
    T t = T(2.0 / OF_K23) * temp * y2;                  // Eq. (tred)
    T dtdn = T(-2.0 / 3.0) * t * rn;
    T tf[8];
    if (fp.kind == 0) {                                 // ftTF: f = tau0 kappa, kappa = xi - zeta
        tfunc_eval<T, 2>(tab, t, tf);
        T xi = tf[0], ze = tf[1], dxi = tf[4], dze = tf[5];
        o.f = tau0 * (xi - ze);
        o.ts = tau0 * ze;
        o.dfdn = dtau0 * (xi - ze) + tau0 * (dxi - dze) * dtdn;   // Eq. (vTF)
        o.wc = T(0);
        return o;
    }
    tfunc_eval<T>(tab, t, tf);
    T xi = tf[0], ze = tf[1], A = tf[2], B = tf[3];
    T dxi = tf[4], dze = tf[5], dA = tf[6], dB = tf[7];
    // s^2 = |grad n|^2 / (4 (3 pi^2)^{2/3} n^{8/3})  (Eq. (s_0defn))
    T rn43 = rn * y;
    T s2 = (g2 * rn43) * rn43 * T(OF_CS);               // ordered so n^{-8/3} never forms alone
    T xt = s2 * A, xs = s2 * B;                          // s_tau^2, s_sigma^2 (Eq. (s_s))
    T Ft, dFt, Fsg, dFsg;
    enhance<T>(fp, xt, Ft, dFt);
    enhance<T>(fp, xs, Fsg, dFsg);
    T Fs = T(2) - Fsg, dFs = -dFsg;                      // F_sigma = 2 - F_tau(s_sigma)
    T kin = tau0 * xi, ent = tau0 * ze;
    o.f = kin * Ft - ent * Fs;                           // Eq. (FGGA)
    o.ts = ent * Fs;
    T e83 = T(-8.0 / 3.0) * rn;
    // Eq. (vftGGA), first two lines (every sigma term carries the minus sign of Eq. (FGGA))
    o.dfdn = dtau0 * (xi * Ft - ze * Fs) + tau0 * dtdn * (dxi * Ft - dze * Fs)
             + kin * dFt * (e83 * xt + s2 * dA * dtdn)
             - ent * dFs * (e83 * xs + s2 * dB * dtdn);
    // last line: W = [tau0 xi F_tau' A - tau0 zeta F_sigma' B] d s^2/d grad n
    o.wc = ((kin * dFt * A - ent * dFs * B) * rn43) * rn43 * T(2 * OF_CS);
    return o;
}

// Perdew-Zunger 1981 unpolarised LDA: eps_xc and v_xc = eps_xc - (r_s/3) d eps_xc/d r_s.
// gamma, beta1, beta2, A, B as published; C and D are fixed by continuity of
// eps_c and its r_s derivative at r_s = 1 (the published rounded C, D leave a
// small jump there).
constexpr double kPzDen = 1.0 + 1.0529 + 0.3334;
constexpr double kPzD = -0.1423 / kPzDen + 0.048;                                // B + D = eps_pade(1)
constexpr double kPzC = 0.1423 * (0.5 * 1.0529 + 0.3334) / (kPzDen * kPzDen) - 0.0311 - kPzD;

// y = n^{-1/3} as computed by the caller.
template <typename T>
OF_HD void pz81_point(T n, T y, T &eps, T &v)
{
    T rs = T(0.62035049089940001667) * y;              // (3/(4 pi n))^{1/3}
    T ex = T(-0.73855876638202240587) * n * y * y;     // -(3/4)(3/pi)^{1/3} n^{1/3}
    T ec, vc;
    if (rs >= T(1)) {
        T sq = sqrt(rs);
        T den = T(1) / (T(1) + T(1.0529) * sq + T(0.3334) * rs);
        ec = T(-0.1423) * den;
        vc = ec * (T(1) + T(7.0 / 6.0 * 1.0529) * sq + T(4.0 / 3.0 * 0.3334) * rs) * den;
    } else {
        T lr = log(rs);
        ec = T(0.0311) * lr + T(-0.048) + T(kPzC) * rs * lr + T(kPzD) * rs;
        vc = T(0.0311) * lr + T(-0.048 - 0.0311 / 3.0) + T(2.0 / 3.0 * kPzC) * rs * lr
             + T((2.0 * kPzD - kPzC) / 3.0) * rs;
    }
    eps = ex + ec;
    v = T(4.0 / 3.0) * ex + vc;
}

template <typename T>
OF_HD void pz81_point(T n, T &eps, T &v)
{
    pz81_point<T>(n, inv_cbrt(n), eps, v);
}

// ---------------------------------------------------------------------------
// The same pointwise functional in double-float arithmetic (ffmath.cuh) for
// the FP64 path's double-float kernels: every intermediate is a double-float,
// so the result agrees with the binary64 routines above to about 1e-13 of the
// size of its terms while running on the FP32 units.  Outside the domain
// below (and in the Sommerfeld and classical branches of the temperature
// functions) pw_core_f2 returns false and the caller uses binary64.  The
// split table (hi, lo per coefficient) follows the binary64 one.

template <typename T> struct PwOut {
    T f, ts, dfdn, wc, eps, vxc;
};

constexpr double kPwNmin = 1e-18, kPwNmax = 1e18, kPwS2max = 1e10;

// The double-float Horner evaluations run several polynomials side by side
// (the four temperature functions; the enhancement factor at both of its
// arguments): one rolled loop over the degree, so that the code stays small
// (instruction fetch) and the chains of one warp overlap.  Each polynomial
// comes with its derivative dp and half its second derivative d2 at the
// binary32 panel variable; the terms of degree >= split are summed in
// binary32: their sum, times u^split, is below 2^-24 of the scale the
// polynomial enters with on every panel, so binary32 rounding there stays
// below the double-float rounding.
struct HornerF2 {
    ff::f2 p, dp;   // unnormalised
    float d2;
};
OF_HD void horner_lo(HornerF2 &h, float u, float c)
{
    h.d2 = h.d2 * u + h.dp.hi;
    h.dp.hi = h.dp.hi * u + h.p.hi;
    h.p.hi = h.p.hi * u + c;
}
OF_HD void horner_dd(HornerF2 &h, float u, ff::f2 c)
{
    h.d2 = h.d2 * u + h.dp.hi;
    h.dp = ff::fma_step_u(h.dp, u, h.p);
    h.p = ff::fma_step_u(h.p, u, c);
}

// The step from a binary32 tail to its first pair: the derivative, one degree
// behind, stays in binary32.
OF_HD void horner_first(HornerF2 &h, float u, ff::f2 c)
{
    h.d2 = h.d2 * u + h.dp.hi;
    h.dp.hi = h.dp.hi * u + h.p.hi;
    const ff::f2 m = ff::two_prod(h.p.hi, u), s = ff::two_sum(m.hi, c.hi);
    h.p = ff::f2(s.hi, ff::fadd(m.lo, ff::fadd(s.lo, c.lo)));
}

// Table polynomials with the refined double-float table (kTfDdSub panels an
// octave).  The panel variable u = uh + ul: uh is exact in binary32 and the
// Horner sums run with it; ul (below 2e-6) enters through the first and
// second derivatives.  The tails in binary32 (degrees 6 to 10) cost, over
// every panel, at most 8e-19 of xi, 2e-18 of xi for zeta (zeta comes close to
// zero but enters only beside xi, f = tau0 xi F_tau - tau0 zeta F_sigma),
// 5e-17 of A and 8e-17 of the larger of B and A xi / zeta (B enters through
// zeta F(s^2 B) beside xi F(s^2 A)); of the derivatives per ln t, which the
// potential takes, 2e-16, 3e-16, 9e-15 and 1.6e-14.  (From degree 5 up in
// binary32 and without degree 10, A and B put 9.6e-13 into df/dn where s^2 is
// large.)  With the unrefined panels 7, 7, 8 and all 10 degrees needed
// double-float: 32 steps instead of 24.
template <int NF>
OF_HD void tfunc_eval_f2(const ff::f2 *__restrict__ tab, ff::f2 t, ff::f2 out[8])
{
    static_assert(kTfFuncs == 4 && (NF == 2 || NF == 4), "rows of four functions");
    int e;
    float inv2e;
    const float m = split_pow2(t.hi, e, inv2e);
    const int sub = (int)((m - 1.0f) * (float)kTfDdSub);
    const float uh = (float)(2 * kTfDdSub) * (m - 1.0f) - (float)(2 * sub + 1);
    const float ul = (float)(2 * kTfDdSub) * t.lo * inv2e;
    const float dudt = (float)(2 * kTfDdSub) * inv2e;
    const float4 *c = reinterpret_cast<const float4 *>(tab + (size_t)((e - kTfEmin) * kTfDdSub + sub) * kTfDdRow);
    const float4 *tail = c + 2 * kTfSplit;               // tail[k]: degree kTfSplit + k
    HornerF2 h[NF];
    const float4 top = tail[kTfDeg - kTfSplit];
    h[0].p.hi = top.x;
    h[1].p.hi = top.y;
    if (NF == 4) {
        h[2].p.hi = top.z;
        h[3].p.hi = top.w;
    }
#pragma unroll
    for (int q = 0; q < NF; ++q) {
        h[q].p.lo = 0.0f;
        h[q].dp = ff::f2(0.0f, 0.0f);
        h[q].d2 = 0.0f;
    }
#pragma unroll 1
    for (int j = kTfDeg - kTfSplit - 1; j >= 0; --j) {
        const float4 a = tail[j];
        const float cj[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int q = 0; q < NF; ++q) horner_lo(h[q], uh, cj[q]);
    }
    {
        const float4 a = c[2 * kTfSplit - 2];
        horner_first(h[0], uh, ff::f2(a.x, a.y));
        horner_first(h[1], uh, ff::f2(a.z, a.w));
        if (NF == 4) {
            const float4 b = c[2 * kTfSplit - 1];
            horner_first(h[2], uh, ff::f2(b.x, b.y));
            horner_first(h[3], uh, ff::f2(b.z, b.w));
        }
    }
#pragma unroll 1
    for (int j = kTfSplit - 2; j >= 0; --j) {
        const float4 a = c[2 * j];
        horner_dd(h[0], uh, ff::f2(a.x, a.y));
        horner_dd(h[1], uh, ff::f2(a.z, a.w));
        if (NF == 4) {
            const float4 b = c[2 * j + 1];
            horner_dd(h[2], uh, ff::f2(b.x, b.y));
            horner_dd(h[3], uh, ff::f2(b.z, b.w));
        }
    }
#pragma unroll
    for (int q = 0; q < NF; ++q) {
        // normalised first: the sums round at the size of the low words
        const ff::f2 p = ff::fast_two_sum(h[q].p.hi, h[q].p.lo), dp = ff::fast_two_sum(h[q].dp.hi, h[q].dp.lo);
        out[q] = ff::add(p, dp.hi * ul);
        out[4 + q] = ff::scale(ff::add(dp, 2.0f * h[q].d2 * ul), dudt);
    }
}

// Enhancement factor F(x) and dF/dx in double-float (forms as in enhance).
FF_CALL void enhance_f2(const FuncParams &fp, ff::f2 x, ff::f2 &F, ff::f2 &dF)
{
    using namespace ff;
    if (fp.kind == 1) {                                     // SGA form
        const f2 p0 = from_double(fp.p0);
        F = add(mul(x, p0), 1.0f);
        dF = p0;
    } else if (fp.kind == 3) {                              // KST2 form
        const f2 p0 = from_double(fp.p0), p1 = from_double(fp.p1);
        f2 den = recip(add(mul(x, p1), 1.0f));
        F = add(mul(mul(x, p0), den), 1.0f);
        dF = mul(p0, mul(den, den));
    } else {                                                // VT84F, m = 8, n = 4
        const f2 mu = FFC(2.778), al = FFC(1.2965);
        if (x.hi <= 1e-15f) {                               // F = 1 + O(x)
            F = {1.0f, 0.0f};
            dF = FFC(-2.778 + 1.2965 + 5.0 / 3.0);
            return;
        }
        const f2 ax = mul(x, al);
        const f2 e1 = exp(neg(ax));                         // e^(-al x)
        const f2 x2 = mul(x, x);
        const f2 em = neg(expm1_neg(neg(mul(x2, al))));     // 1 - e^(-al x^2)
        const f2 mx = mul(x, mu);
        const f2 q = add(mx, 1.0f);                         // 1 + mu x
        const f2 inv = recip(mul(x, q));
        const f2 rx = mul(q, inv);                          // 1/x
        const f2 den = mul(x, inv);                         // 1/(1 + mu x)
        // F = 1 - mu x e1 den + em (rx - 1) + (5/3) x
        f2 Fv = add(neg(mul(mul(mx, e1), den)), 1.0f);
        Fv = add(Fv, mul(em, add(rx, -1.0f)));
        F = add(Fv, mul(x, FFC(5.0 / 3.0)));
        // dF = -mu e1 (1 - al x - al mu x^2) den^2 + 2 al (1 - em)(1 - x) - em rx^2 + 5/3
        const f2 poly = add(neg(add(ax, mul(mul(x2, al), mu))), 1.0f);
        f2 d = neg(mul(mul(mul(mu, e1), poly), mul(den, den)));
        d = add(d, mul(mul(al, add(neg(em), 1.0f)), scale(add(neg(x), 1.0f), 2.0f)));
        d = sub(d, mul(em, mul(rx, rx)));
        dF = add(d, FFC(5.0 / 3.0));
    }
}

// VT84F F(x) and dF/dx in double-float outside the enhancement table's
// range: x < 2^-20: the cubic series (the next terms are below 1e-16 in F
// and dF), x >= 64: F = 5x/3 + 1/x.
FF_CALL void enhance_vt84f_ends(ff::f2 x, ff::f2 &F, ff::f2 &dF)
{
    using namespace ff;
    if (x.hi < 9.5367431640625e-07f) {
        // series of Eq. (VT84F): c1 = alpha - mu + 5/3, c2 = mu (alpha + mu) - alpha,
        // c3 = -mu (alpha^2/2 + alpha mu + mu^2) - alpha^2/2 (the x^3 term matters
        // for dF at the 1e-12 level)
        constexpr double mu = 2.778, al = 1.2965;
        constexpr double c1 = al - mu + 5.0 / 3.0, c2 = mu * (al + mu) - al;
        constexpr double c3 = -mu * (0.5 * al * al + al * mu + mu * mu) - 0.5 * al * al;
        F = add(mul(x, add(mul(x, add(mul(x, FFC(c3)), FFC(c2))), FFC(c1))), 1.0f);
        dF = add(mul(x, add(mul(x, FFC(3.0 * c3)), FFC(2.0 * c2))), FFC(c1));
        return;
    }
    const f2 r = recip(x);
    F = add(mul(x, FFC(5.0 / 3.0)), r);
    dF = sub(FFC(5.0 / 3.0), mul(r, r));
}

// VT84F F and dF/dx at two arguments from the enhancement table etab of
// G = (F - 1)/x: F = 1 + x G, dF = G + x G' with G' the polynomial's
// derivative, so the potential is the exact derivative of the tabulated
// energy.  (Tail of G from degree kEnSplit up: 1.3e-8.)
OF_HD void enhance_vt84f_tab(const ff::f2 *__restrict__ etab, const ff::f2 (&x)[2], ff::f2 (&F)[2], ff::f2 (&dF)[2])
{
    using namespace ff;
    float uh[2], ul[2], dudx[2];
    const float4 *c[2];
    bool in[2];
    HornerF2 h[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        in[k] = x[k].hi >= 9.5367431640625e-07f && x[k].hi < 64.0f;
        int e;
        float inv2e;
        const float m = split_pow2(in[k] ? x[k].hi : 1.0f, e, inv2e);
        const int sub = (int)((m - 1.0f) * (float)kEnSub);
        uh[k] = (float)(2 * kEnSub) * (m - 1.0f) - (float)(2 * sub + 1);
        ul[k] = (float)(2 * kEnSub) * x[k].lo * inv2e;
        dudx[k] = (float)(2 * kEnSub) * inv2e;
        c[k] = reinterpret_cast<const float4 *>(etab + (size_t)((e - kEnEmin) * kEnSub + sub) * kEnDdRow);
        const float4 a = c[k][3], b = c[k][4];   // degrees 5 .. 8, 9 and 10
        h[k] = {{b.y, 0.0f}, {0.0f, 0.0f}, 0.0f};
        horner_lo(h[k], uh[k], b.x);
        horner_lo(h[k], uh[k], a.w);
        horner_lo(h[k], uh[k], a.z);
        horner_lo(h[k], uh[k], a.y);
        horner_lo(h[k], uh[k], a.x);
        horner_dd(h[k], uh[k], f2(c[k][2].x, c[k][2].y));   // degree 4
    }
#pragma unroll 1
    for (int j = 1; j >= 0; --j)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const float4 a = c[k][j];            // degrees 2 j, 2 j + 1
            horner_dd(h[k], uh[k], f2(a.z, a.w));
            horner_dd(h[k], uh[k], f2(a.x, a.y));
        }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const f2 G = add(h[k].p, h[k].dp.hi * ul[k]);
        const f2 dG = scale(add(h[k].dp, 2.0f * h[k].d2 * ul[k]), dudx[k]);
        F[k] = add(mul(x[k], G), 1.0f);
        dF[k] = add_s(G, mul(x[k], dG));
    }
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if (!in[k]) enhance_vt84f_ends(x[k], F[k], dF[k]);
}

// ln x for x > 0 (normal binary32 range): x = 2^e m, the table's binary32
// reciprocal r of the centre of m's 2^-8-wide interval and its -ln r, then
// ln m = -ln r + log1p(m r - 1) with |m r - 1| < 2^-8.9: the square in
// double-float, the terms from the cube on in binary32.  Absolute error a
// few 2^-48 max(1, |ln x|).
OF_HD ff::f2 log_tab(const ff::f2 *__restrict__ ltab, ff::f2 x)
{
    using namespace ff;
    int e;
    float inv2e;
    const float m = split_pow2(x.hi, e, inv2e);
    const int i = (int)((m - 1.0f) * (float)kLgSub);
    const float r = ltab[2 * i].hi;
    const f2 z = two_prod(m, r);
    const f2 d = add(f2(fadd(z.hi, -1.0f), z.lo), fmul(fmul(x.lo, inv2e), r));   // z.hi - 1 is exact
    const float t = d.hi;
    const f2 sq = two_prod(t, t);
    const float cube = fmul(t * t, t) * (1.0f / 3.0f + t * (-0.25f + t * (0.2f - t * (1.0f / 6.0f))));
    const f2 l1 = add(d, f2(-0.5f * sq.hi, ffma(-t, d.lo, -0.5f * sq.lo) + cube));
    const f2 k = two_prod((float)e, FFC(kLn2).hi);
    const f2 base = add(f2(k.hi, ffma((float)e, FFC(kLn2).lo, k.lo)), ltab[2 * i + 1]);
    return add(base, l1);
}

// PZ81 (same branches and constants as pz81_point) from n, n^(1/3) and
// y = n^(-1/3) in double-float.  Sums of like terms of one size: add_s.
OF_HD void pz81_f2(const ff::f2 *__restrict__ ltab, ff::f2 c13, ff::f2 y, ff::f2 &eps, ff::f2 &v)
{
    using namespace ff;
    const f2 rs = mul(y, FFC(0.62035049089940001667));
    const f2 ex = mul(c13, FFC(-0.73855876638202240587));
    f2 ec, vc;
    if (rs.hi >= 1.0f) {
        const f2 sq = sqrt(rs);
        const f2 den = recip(add(add_s(mul(sq, FFC(1.0529)), mul(rs, FFC(0.3334))), 1.0f));
        ec = mul(den, FFC(-0.1423));
        const f2 num = add(add_s(mul(sq, FFC(7.0 / 6.0 * 1.0529)), mul(rs, FFC(4.0 / 3.0 * 0.3334))), 1.0f);
        vc = mul(mul(ec, num), den);
    } else {
        const f2 lr = log_tab(ltab, rs);
        const f2 rlr = mul(rs, lr), al = mul(lr, FFC(0.0311));
        ec = add_s(add_s(al, FFC(-0.048)), add_s(mul(rlr, FFC(kPzC)), mul(rs, FFC(kPzD))));
        vc = add_s(add_s(al, FFC(-0.048 - 0.0311 / 3.0)),
                   add_s(mul(rlr, FFC(2.0 / 3.0 * kPzC)), mul(rs, FFC((2.0 * kPzD - kPzC) / 3.0))));
    }
    eps = add_s(ex, ec);
    v = add_s(mul(ex, FFC(4.0 / 3.0)), vc);
}

// Double-float outputs of the pointwise functional at one point.
struct PwF2 {
    ff::f2 f, ts, dfdn, eps, vxc;
    ff::f2 w[3];    // W = d f_s / d(grad n), by component
    ff::f2 wg;      // W . grad n
};

// f_s, its derivatives and (xc != 0) PZ81 at one point from n and the
// gradient components gr[3] in double-float; false when the point is
// outside the double-float domain (s^2 is formed from (grad n) n^(-4/3), so
// an s^2 past kPwS2max, or one that overflows, also returns false).
// tcoef = 2 k_B T / (3 pi^2)^(2/3).
OF_HD bool pw_core_f2(const FuncParams &fp, const ff::f2 *__restrict__ tab, ff::f2 tcoef, ff::f2 n,
                      const ff::f2 *gr, int xc, PwF2 &o)
{
    using namespace ff;
    if (!(n.hi >= (float)kPwNmin && n.hi <= (float)kPwNmax)) return false;
    const f2 y = rcbrt(n);                                   // n^(-1/3)
    const f2 y2 = mul(y, y);
    const f2 t = mul(tcoef, y2);                             // Eq. (tred)
    if (!(t.hi >= 9.5367431640625e-07f && t.hi < 17179869184.0f)) return false;
    const f2 c13 = mul(n, y2);                               // n^(1/3)
    const f2 n23 = mul(c13, c13);
    const f2 rn = mul(y2, y);                                // 1/n
    const f2 tau0 = mul(mul(n, n23), FFC(OF_CTF));           // Eq. (tauTFdefn)
    const f2 dtdn = mul(mul(t, rn), FFC(-2.0 / 3.0));
    f2 tf[8];
    if (fp.kind == 0) {                                      // ftTF
        tfunc_eval_f2<2>(tab, t, tf);
        const f2 kap = sub(tf[0], tf[1]);
        o.f = mul(tau0, kap);
        o.ts = mul(tau0, tf[1]);
        const f2 dtau0 = mul(n23, FFC(5.0 / 3.0 * OF_CTF));
        o.dfdn = add(mul(dtau0, kap), mul(mul(tau0, sub(tf[4], tf[5])), dtdn));   // Eq. (vTF)
        o.w[0] = o.w[1] = o.w[2] = o.wg = f2(0.0f, 0.0f);
    } else {
        const f2 rn43 = mul(y2, y2);                         // n^(-4/3)
        const f2 q0 = mul(gr[0], rn43), q1 = mul(gr[1], rn43), q2 = mul(gr[2], rn43);
        const f2 s2 = mul(add_s(add_s(mul(q0, q0), mul(q1, q1)), mul(q2, q2)), FFC(OF_CS));   // Eq. (s_0defn)
        if (!(s2.hi <= (float)kPwS2max)) return false;
        tfunc_eval_f2<4>(tab, t, tf);
        const f2 xi = tf[0], ze = tf[1], A = tf[2], B = tf[3];
        const f2 dxi = tf[4], dze = tf[5], dA = tf[6], dB = tf[7];
        const f2 xt = mul(s2, A), xs = mul(s2, B);           // Eq. (s_s)
        f2 Ft, dFt, Fsg, dFsg;
        if (fp.kind == 2) {                                  // VT84F: the enhancement table
            const f2 *etab = tab + kTfDdSize;
            const f2 xx[2] = {xt, xs};
            f2 FF[2], dFF[2];
            enhance_vt84f_tab(etab, xx, FF, dFF);
            Ft = FF[0], dFt = dFF[0], Fsg = FF[1], dFsg = dFF[1];
        } else {
            enhance_f2(fp, xt, Ft, dFt);
            enhance_f2(fp, xs, Fsg, dFsg);
        }
        const f2 Fs = add(neg(Fsg), 2.0f), dFs = neg(dFsg); // F_sigma = 2 - F_tau(s_sigma)
        const f2 kin = mul(tau0, xi), ent = mul(tau0, ze);
        // (add_s below: the operands carry a few u^2 of their own size, and
        // every sum is judged against the size of its terms)
        const f2 eF = mul(ent, Fs);
        o.f = add_s(mul(kin, Ft), neg(eF));                 // Eq. (FGGA)
        o.ts = eF;
        const f2 e83 = mul(rn, FFC(-8.0 / 3.0));
        const f2 s2dt = mul(s2, dtdn);
        const f2 kF = mul(kin, dFt), sF = mul(ent, dFs);
        // Eq. (vftGGA), first two lines; dtau0 (xi F_tau - zeta F_sigma) = (5/3) f / n
        f2 d = mul(div(o.f, n), FFC(5.0 / 3.0));
        d = add_s(d, mul(mul(tau0, dtdn), add_s(mul(dxi, Ft), neg(mul(dze, Fs)))));
        d = add_s(d, mul(kF, add_s(mul(e83, xt), mul(s2dt, dA))));
        d = add_s(d, neg(mul(sF, add_s(mul(e83, xs), mul(s2dt, dB)))));
        o.dfdn = d;
        // last line: W = [tau0 xi F_tau' A - tau0 zeta F_sigma' B] d s^2 / d grad n
        const f2 wpre = add_s(mul(kF, A), neg(mul(sF, B)));
        const f2 wr = mul(mul(wpre, rn43), FFC(2.0 * OF_CS));
        o.w[0] = mul(wr, q0);
        o.w[1] = mul(wr, q1);
        o.w[2] = mul(wr, q2);
        o.wg = scale(mul(wpre, s2), 2.0f);                  // d s^2/d grad n . grad n = 2 s^2
    }
    if (xc) {
        pz81_f2(tab + kTfDdSize + kEnDdSize, c13, y, o.eps, o.vxc);
    } else {
        o.eps = f2(0.0f, 0.0f);
        o.vxc = f2(0.0f, 0.0f);
    }
    return true;
}

// The routines of the precision T (binary64 or binary32) with the same output.
template <typename T>
OF_HD PwOut<T> pw_point_native(const FuncParams &fp, const T *__restrict__ tab, T temp, T n, T g2, int xc)
{
    FsOut<T> s = fs_point<T>(fp, tab, temp, n, g2);
    PwOut<T> o;
    o.f = s.f;
    o.ts = s.ts;
    o.dfdn = s.dfdn;
    o.wc = s.wc;
    o.eps = T(0);
    o.vxc = T(0);
    if (xc) pz81_point<T>(n, s.y13, o.eps, o.vxc);
    return o;
}


// The FP64 field sets' tables in dst[kDdTabSize]: the binary64 temperature
// table, its refined double-float copy, the double-float VT84F enhancement
// table and the logarithm table (the last three contiguous, as pw_core_f2
// reads them).
inline void dd_tables_fill(const double *ttab, double *dst)
{
    for (int i = 0; i < kTfSize; ++i) dst[i] = ttab[i];
    float *rf = reinterpret_cast<float *>(dst + kTfSize);
    for (int p = 0; p < kTfPanels; ++p)
        for (int s = 0; s < kTfRef; ++s)
            for (int q = 0; q < kTfFuncs; ++q) {
                // u = ctr + v / kTfRef: Taylor coefficients about ctr by repeated synthetic division
                const double ctr = (2.0 * s + 1.0 - kTfRef) / kTfRef;
                double a[kTfNc], sc = 1.0;
                for (int k = 0; k < kTfNc; ++k) a[k] = ttab[((size_t)p * kTfFuncs + q) * kTfNc + k];
                for (int k = 0; k < kTfDeg; ++k)
                    for (int j = kTfDeg - 1; j >= k; --j) a[j] += ctr * a[j + 1];
                float *row = rf + 2 * (size_t)(p * kTfRef + s) * kTfDdRow;
                for (int k = 0; k <= kTfDeg; ++k, sc /= kTfRef) {
                    const ff::f2 c = ff::from_double(a[k] * sc);
                    if (k < kTfSplit) {
                        row[2 * (k * kTfFuncs + q)] = c.hi;
                        row[2 * (k * kTfFuncs + q) + 1] = c.lo;
                    } else {
                        row[2 * kTfSplit * kTfFuncs + (k - kTfSplit) * kTfFuncs + q] = c.hi;
                    }
                }
            }
    float *en = reinterpret_cast<float *>(dst + kTfSize + kTfDdSize);
    double etab[kEnSize];
    enh_table_fill(etab);
    for (int p = 0; p < kEnPanels; ++p) {
        float *row = en + 2 * (size_t)p * kEnDdRow;
        for (int k = 0; k < 2 * kEnDdRow; ++k) row[k] = 0.0f;
        for (int k = 0; k < kEnNc; ++k) {
            const ff::f2 c = ff::from_double(etab[(size_t)p * kEnNc + k]);
            if (k < kEnSplit) {
                row[2 * k] = c.hi;
                row[2 * k + 1] = c.lo;
            } else {
                row[(kEnSplit + 1) / 2 * 4 + k - kEnSplit] = c.hi;
            }
        }
    }
    float *lg = en + 2 * kEnDdSize;   // {r, 0}, -ln r per interval
    for (int i = 0; i < kLgSub; ++i) {
        const float r = (float)(1.0 / (1.0 + (i + 0.5) / kLgSub));
        const long double l = -logl((long double)r);
        lg[4 * i] = r;
        lg[4 * i + 1] = 0.0f;
        lg[4 * i + 2] = (float)l;
        lg[4 * i + 3] = (float)(l - (long double)(float)l);
    }
}

}  // namespace ofdft
