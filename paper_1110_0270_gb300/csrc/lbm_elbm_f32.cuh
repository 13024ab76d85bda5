// ELBM (Section 3) for FP32 arithmetic (FP32 and 16-bit storage) on the FP32
// pipe: f* - f and the root of S(f + alpha (f* - f)) = S(f) in double-single
// arithmetic (an unevaluated sum h + l of two floats, about 47 bits).
//
// Why: a GB300 SM finishes one FP64 warp instruction in 19 clocks (measured,
// any mix of add, mul and fma) against about a third of a clock for FP32, so
// the FP64 form of this step (100 FP64 instructions near rest, about 1,000
// where alpha is solved) is bound by the FP64 pipe at 3-5% of the HBM rate.
// The double-single form runs on the FP32 pipe instead.
//
// What is kept in two floats: rho, rho u, u, the equilibrium, f* - f and the
// two leading moments of the root equation; the higher orders of that
// equation enter as small corrections and are FP32 sums.  Sites outside the
// range the error bounds below hold for (kFf* constants) take the FP64 solve.
#pragma once

#include "lbm_elbm_lanes.cuh"

namespace lbm {

// Correctly rounded single operations that are neither contracted nor
// reassociated (the error terms below depend on it).
__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float ffma(float a, float b, float c) { return __fmaf_rn(a, b, c); }

struct Ff {
    float h, l;
};

// a + b = s.h + s.l exactly (Knuth's two-sum).
__device__ __forceinline__ Ff two_sum(float a, float b) {
    const float s = fadd(a, b), t = fsub(s, a);
    return {s, fadd(fsub(a, fsub(s, t)), fsub(b, t))};
}
// The same for |a| >= |b| (Dekker's fast two-sum).
__device__ __forceinline__ Ff fast_two_sum(float a, float b) {
    const float s = fadd(a, b);
    return {s, fsub(b, fsub(s, a))};
}
// a + b for double-single a, b of any order.
__device__ __forceinline__ Ff ff_add(Ff a, Ff b) {
    const Ff s = two_sum(a.h, b.h);
    return fast_two_sum(s.h, fadd(s.l, fadd(a.l, b.l)));
}
// a b, the low part not folded into the high one.
__device__ __forceinline__ Ff ff_mul(Ff a, Ff b) {
    const float p = fmul(a.h, b.h);
    return {p, ffma(a.l, b.h, ffma(a.h, b.l, ffma(a.h, b.h, -p)))};
}

// The range of the FP32 forms: a density for which no error term is
// subnormal, a velocity for which ff_axis meets fast_two_sum's order with
// positive factors (u / 2 below a = 1/6 + ...), and, with x_i =
// (f*_i - f_i) / f*_i, for the short form |x| < 1/4 up to |u| = 0.2 and
// |x| < 1/16 up to 0.4, which keep the rest population above every other one
// (the order of rho's partial sums) and f* within a factor 2 of f.
constexpr float kFfRhoMin = 0x1p-20f, kFfRhoMax = 0x1p20f, kFfUMax = 0.4f;
__device__ __forceinline__ float ff_x_limit(float ux, float uy) {
    const float u = fmaxf(fabsf(ux), fabsf(uy));
    return u <= 0.2f ? 0.25f : (u <= kFfUMax ? 0.0625f : 0.f);
}

// One site's entropic state: density, velocity, and f* - f = Dh + Dl per
// population, where f* = (Dh + f) + Dl, both sums exact: with |x| < 1/4 the
// high part of f* lies within a factor 2 of f, so their difference is exact
// (Sterbenz).  f* - f is within 2^-41 f* of its exact value (measured against
// quad precision: 2^-41.5 over |u| <= 0.2, 2^-40.1 over |u| <= 0.4).
template <int Q>
struct FfSite {
    float rho, ux, uy;
    float Dh[Q], Dl[Q];
};

// 1D entropic factors a - u/2, 1 - 2a, a + u/2 with a = (2 sqrt(1 + 3 u^2) - 1) / 6.
__device__ __forceinline__ void ff_axis(Ff u, Ff* ax) {
    // t = 1 + 3 u^2
    const float p = fmul(u.h, u.h), q = fmul(3.f, p);
    const float pe = ffma(fadd(u.h, u.h), u.l, ffma(u.h, u.h, -p));
    Ff t = fast_two_sum(1.f, q);
    t.l = fadd(t.l, ffma(3.f, pe, ffma(3.f, p, -q)));
    // s + sl = sqrt(t): a Newton step to the rounded root of t.h, one more
    // for its low part
    const float rs = rsqrtf(t.h), hs = fmul(0.5f, rs), s0 = fmul(t.h, rs);
    const float s = ffma(hs, ffma(-s0, s0, t.h), s0);
    const float sl = fmul(hs, fadd(ffma(-s, s, t.h), t.l));
    // a = s / 3 - 1 / 6
    constexpr float c3 = (float)(1.0 / 3.0), c3l = (float)(1.0 / 3.0 - (double)c3);
    constexpr float c6 = (float)(1.0 / 6.0), c6l = (float)(1.0 / 6.0 - (double)c6);
    const float w = fmul(s, c3);
    Ff a = fast_two_sum(w, -c6);
    a.l = fadd(a.l, fsub(ffma(sl, c3, ffma(s, c3l, ffma(s, c3, -w))), c6l));
    const float uh = fmul(0.5f, u.h), ul = fmul(0.5f, u.l);
    ax[0] = fast_two_sum(a.h, -uh);
    ax[0].l = fadd(ax[0].l, fsub(a.l, ul));
    ax[2] = fast_two_sum(a.h, uh);
    ax[2].l = fadd(ax[2].l, fadd(a.l, ul));
    ax[1] = fast_two_sum(1.f, fmul(-2.f, a.h));
    ax[1].l = ffma(-2.f, a.l, ax[1].l);
}

// FAR: populations of any order and distance from f* (exact sums of any order).
template <int Q, bool FAR>
__device__ __forceinline__ void ff_site(const float* f, FfSite<Q>& s) {
    using L = Lat<Q>;
    // rho: from the largest population (the rest one) on, so that each
    // partial sum is at least the next term
    Ff rho = {f[L::rest], 0.f};
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        if (i == L::rest) continue;
        const Ff t = FAR ? two_sum(rho.h, f[i]) : fast_two_sum(rho.h, f[i]);
        rho = {t.h, fadd(rho.l, t.l)};
    }
    rho = fast_two_sum(rho.h, rho.l);
    // rho u from the differences of opposite populations
    Ff jx = {0.f, 0.f}, jy = {0.f, 0.f};
    bool fx = true, fy = true;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int o = L::opp(i);
        if (o <= i) continue;
        const Ff d = two_sum(f[i], -f[o]);
        if (L::cx(i) != 0) {
            const Ff e = L::cx(i) > 0 ? d : Ff{-d.h, -d.l};
            if (fx) {
                jx = e;
            } else {
                const Ff t = two_sum(jx.h, e.h);
                jx = {t.h, fadd(t.l, fadd(jx.l, e.l))};
            }
            fx = false;
        }
        if (L::cy(i) != 0) {
            const Ff e = L::cy(i) > 0 ? d : Ff{-d.h, -d.l};
            if (fy) {
                jy = e;
            } else {
                const Ff t = two_sum(jy.h, e.h);
                jy = {t.h, fadd(t.l, fadd(jy.l, e.l))};
            }
            fy = false;
        }
    }
    // 1 / rho = r + r (e + e^2), e = 1 - rho r
    const float r = __fdividef(1.f, rho.h);
    const float e = ffma(-rho.l, r, ffma(-rho.h, r, 1.f));
    const Ff inv = {r, fmul(r, ffma(e, e, e))};
    Ff u = ff_mul(jx, inv), ax[3], ay[3];
    u = fast_two_sum(u.h, u.l);
    s.rho = rho.h;
    s.ux = u.h;
    s.uy = 0.f;
    ff_axis(u, ax);
#pragma unroll
    for (int k = 0; k < 3; ++k) ax[k] = ff_mul(rho, ax[k]);
    if (Q == 9) {
        u = ff_mul(jy, inv);
        u = fast_two_sum(u.h, u.l);
        s.uy = u.h;
        ff_axis(u, ay);
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const Ff fe = Q == 9 ? ff_mul(ax[L::cx(i) + 1], ay[L::cy(i) + 1]) : ax[L::cx(i) + 1];
        if (FAR) {
            const Ff d = two_sum(fe.h, -f[i]);
            s.Dh[i] = d.h;
            s.Dl[i] = fadd(d.l, fe.l);
        } else {
            s.Dh[i] = fsub(fe.h, f[i]);
            s.Dl[i] = fe.l;
        }
    }
}

// The root.  With d_i = (f*_i - f_i) / f*_i, a = alpha - 1 and
// g(x) = (1 + x) ln(1 + x) - x = sum_{n >= 2} c_n x^n, c_n = (-1)^n / (n (n-1)),
//   -S_f(alpha) = sum f*_i [g(a d_i) - g(-d_i)] = sum_n c_n (a^n - (-1)^n) M_n,
// M_n = sum f*_i d_i^n.  In y = alpha - 2 = a - 1, which is of the order of
// d, the two leading orders are y (1 + y / 2) M_2 - (1 + a^3) / 6 M_3, free of
// cancellation; M_2 and M_3 are double-single sums, M_4 ... M_N (a relative
// d^2 of the leading orders) FP32 ones.  Newton's iteration for y runs in
// FP32; its last step takes the residual with the leading orders in
// double-single, which leaves y within a unit in its last place (measured
// against quad precision up to |d| = 1/4: 2^-24 |y|), less than the rounding
// of alpha beta to FP32 that the update takes either way.  The orders left
// out change alpha by at most 2 c_{N+1} max |d|^(N-1) < 2^-36 (the tiers of
// elbm_f32).
// For |d| < 1/4 the root exists: S_f(3) < 0 (g(-d) <= 0.55 d^2 and
// g(2d) >= 1.6 d^2), and alpha_max >= 5.
template <int Q, int N>
__device__ __forceinline__ float ff_root(const float* f, const FfSite<Q>& s) {
    Ff M2 = {0.f, 0.f}, M3 = {0.f, 0.f};
    float M[N + 1];
#pragma unroll
    for (int n = 4; n <= N; ++n) M[n] = 0.f;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const Ff fe = {fadd(s.Dh[i], f[i]), s.Dl[i]};
        const Ff D = fast_two_sum(s.Dh[i], s.Dl[i]);
        const float r = __fdividef(1.f, fe.h), q = fmul(D.h, r);
        const Ff d = fast_two_sum(q, fmul(r, ffma(-q, fe.l, fadd(ffma(-q, fe.h, D.h), D.l))));
        const Ff w = ff_mul(D, d);  // f* d^2
        const Ff v = ff_mul(w, d);  // f* d^3
        Ff t = two_sum(M2.h, w.h);
        M2 = {t.h, fadd(M2.l, fadd(t.l, w.l))};
        t = two_sum(M3.h, v.h);
        M3 = {t.h, fadd(M3.l, fadd(t.l, v.l))};
        float z = v.h;
#pragma unroll
        for (int n = 4; n <= N; ++n) {
            z *= d.h;
            M[n] += z;
        }
    }
    M2 = fast_two_sum(M2.h, M2.l);
    M3 = fast_two_sum(M3.h, M3.l);
    const float m2 = M2.h, m3 = M3.h;
    float even = 0.f;  // -sum c_n (-1)^n M_n
#pragma unroll
    for (int n = 4; n <= N; ++n) {
        M[n] *= ((n & 1) ? -1.f : 1.f) / (float)(n * (n - 1));
        even += (n & 1) ? M[n] : -M[n];
    }
    float y = __fdividef(m3, 3.f * m2), tail = 0.f, slope = m2;
    for (int k = 0; k < 8; ++k) {
        const float a = 1.f + y, a2 = a * a;
        float P = M[N], dP = 0.f;  // sum_n c_n M_n a^(n-4) and its derivative
#pragma unroll
        for (int n = N - 1; n >= 4; --n) {
            dP = fmaf(dP, a, P);
            P = fmaf(P, a, M[n]);
        }
        tail = fmaf(a2 * a2, P, even);
        slope = fmaf(m2, a, fmaf(-0.5f * m3, a2, a2 * a * fmaf(a, dP, 4.f * P)));
        const float R = fmaf(m2, y * fmaf(0.5f, y, 1.f),
                             fmaf(-m3, (1.f / 3.f) + (1.f / 6.f) * y * (3.f + y * (3.f + y)), tail));
        const float step = __fdividef(R, slope);
        if (!(fabsf(step) > 1e-6f * fabsf(y))) break;
        y -= step;
    }
    // (tail and slope are those of the last y: the loop leaves before a step
    // of less than 1e-6 y, which moves them by that much)
    constexpr float c3 = (float)(1.0 / 3.0), c3l = (float)(1.0 / 3.0 - (double)c3);
    const float hy = 0.5f * y, yy = fmul(y, hy);
    Ff A = fast_two_sum(y, yy);
    A.l = fadd(A.l, ffma(y, hy, -yy));
    A = ff_mul(M2, A);
    Ff B = fast_two_sum(c3, (1.f / 6.f) * y * (3.f + y * (3.f + y)));
    B.l = fadd(B.l, c3l);
    B = ff_mul(M3, B);
    const Ff t = two_sum(A.h, -B.h);
    const float R = fadd(t.h, fadd(fadd(t.l, fsub(A.l, B.l)), tail));
    return y - __fdividef(R, slope);
}

// The same for |d| < 2^-7 with every moment in FP32 (M2 given): alpha - 2 is
// at most 2^-8 there, so its own relative 2^-21 is 2^-29 of alpha, below the
// rounding of alpha beta to FP32 (measured against quad precision: F is as far
// from exact as from an FP64 alpha).  Two Newton steps from the leading
// order's root (off by a relative d) leave a relative d^4.
template <int Q>
__device__ __forceinline__ float f_root(const FfSite<Q>& s, const float* d, float m2) {
    float m3 = 0.f, m4 = 0.f, m5 = 0.f, m6 = 0.f;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const float v = (s.Dh[i] + s.Dl[i]) * d[i] * d[i], z = v * d[i], zz = z * d[i];
        m3 += v;
        m4 += z;
        m5 += zz;
        m6 = fmaf(zz, d[i], m6);
    }
    // H(y) = m2 y (1 + y/2) - m3 (2 + 3y + 3y^2 + y^3) / 6 + m4 (a^4 - 1) / 12
    //        - m5 (a^5 + 1) / 20 + m6 (a^6 - 1) / 30,  a = 1 + y
    m4 *= 1.f / 12.f;
    m5 *= 1.f / 20.f;
    m6 *= 1.f / 30.f;
    float y = __fdividef(m3, 3.f * m2);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float a = 1.f + y, a2 = a * a, a3 = a2 * a, b = y * (2.f + y);  // b = a^2 - 1
        // even orders from b: a^4 - 1 = b (a^2 + 1), a^6 - 1 = b (a^4 + a^2 + 1)
        const float H = fmaf(m2, y * fmaf(0.5f, y, 1.f),
                             fmaf(-m3, (1.f / 3.f) + (1.f / 6.f) * y * (3.f + y * (3.f + y)),
                                  fmaf(b, fmaf(m4, a2 + 1.f, m6 * fmaf(a2, a2, a2 + 1.f)), -m5 * fmaf(a3, a2, 1.f))));
        const float dH = fmaf(m2, a, fmaf(-0.5f * m3, a2, fmaf(4.f * m4, a3, a2 * a2 * fmaf(6.f * m6, a, -5.f * m5))));
        y -= __fdividef(H, dH);
    }
    return y;
}

template <int Q>
struct ElbmSite {
    float F[Q];
    int code, iters;
};

// F = f + alpha beta (f* - f) from an FP64 solve rounds to FP32 anyway: the
// product in FP32 on the FP64 difference.
template <int Q>
__device__ __forceinline__ void elbm_conserve(const float* f, float* F) {
    float rho, ux, uy;
    moments<Q, float>(f, rho, ux, uy);
    conserve_mass<Q, float>(rho, F);
}

// g(x) and ln(1 + x) (FP32) of a double-single x > -1.  With s = x / (2 + x),
// ln(1 + x) = 2 atanh(s), (2 + x) s = x and T = (atanh(s) - s) / s^3 =
// 1/3 + s^2 T2, T2 = sum_k s^(2k) / (2k + 5): g(x) = x s (1 + (s + s^2) T),
// free of cancellation, for 1/2 <= 1 + x <= 2 (|s| <= 1/3; ten terms leave
// out 2^-36).  Outside, with 1 + x = m 2^e, m in [0.7, 1.42],
// ln(1 + x) = 2 atanh((m - 1) / (m + 1)) + e ln 2 and g = (1 + x) ln(1 + x) - x.
// The leading terms are double-single, T2's part (at most 1% of ln, 0.7% of
// the factor) FP32.
__device__ __forceinline__ Ff ff_div(Ff a, Ff b) {
    const float r = __fdividef(1.f, b.h), q = fmul(a.h, r);
    return fast_two_sum(q, fmul(r, ffma(-q, b.l, fadd(ffma(-q, b.h, a.h), a.l))));
}
__device__ __forceinline__ Ff ff_g(Ff x, float& ln) {
    constexpr float c3 = (float)(1.0 / 3.0), c3l = (float)(1.0 / 3.0 - (double)c3);
    Ff w = two_sum(1.f, x.h);
    w = fast_two_sum(w.h, fadd(w.l, x.l));
    const bool near = w.h >= 0.5f && w.h <= 2.f;
    int e = 0;
    Ff num = x;
    if (!near) {
        // 2^-e w in [0.7, 1.42], less 1: the exponent counts up where the fraction
        // passes that of sqrt(2) (0x3504f3; 0x4afb0d = 2^23 - 0x3504f3)
        e = (int)((__float_as_uint(w.h) + 0x4afb0du) >> 23) - 127;
        const float sc = __uint_as_float((unsigned)(127 - e) << 23);
        num = two_sum(fmul(w.h, sc), -1.f);
        num = fast_two_sum(num.h, fmaf(w.l, sc, num.l));
    }
    Ff den = two_sum(2.f, num.h);
    den.l = fadd(den.l, num.l);
    const Ff s = ff_div(num, den), s2 = ff_mul(s, s);
    const float z = s2.h;
    float t2 = 1.f / 25.f;
#pragma unroll
    for (int k = 9; k >= 0; --k) t2 = fmaf(t2, z, 1.f / (float)(2 * k + 5));
    const float tz = z * t2;
    if (near) {
        ln = 2.f * s.h * fmaf(z, fmaf(z, t2, 1.f / 3.f), 1.f);
        const Ff v = ff_add(s, s2);
        Ff c = ff_mul(v, Ff{c3, c3l});
        c.l = fadd(c.l, fmul(v.h, tz));
        Ff m = two_sum(1.f, c.h);
        m.l = fadd(m.l, c.l);
        const Ff xs = ff_mul(x, s);
        return ff_mul(fast_two_sum(xs.h, xs.l), fast_two_sum(m.h, m.l));
    }
    // atanh(s) = s + s^3 (1/3 + z T2)
    const Ff s3 = ff_mul(s, fast_two_sum(s2.h, s2.l));
    Ff c = ff_mul(s3, Ff{c3, c3l});
    c.l = fadd(c.l, fmul(s3.h, tz));
    const Ff at = ff_add(s, fast_two_sum(c.h, c.l));
    constexpr float l2 = 0.693147180559945309417232121458f;
    constexpr float l2l = (float)(0.693147180559945309417232121458 - (double)l2);
    const Ff k = ff_mul(Ff{(float)e, 0.f}, Ff{l2, l2l});
    const Ff lw = ff_add(Ff{2.f * at.h, 2.f * at.l}, fast_two_sum(k.h, k.l));
    ln = lw.h;
    const Ff wl = ff_mul(w, lw);
    return ff_add(fast_two_sum(wl.h, wl.l), Ff{-x.h, -x.l});
}

// The FP32 solve away from equilibrium (a few sites of a warp at the lid and
// at shocks; on the FP64 path they kept the step of a 257^2 cavity at
// 107 us): |u| < 0.4.  code -1: not settled here, the FP64 solve decides.
// Out of line: its registers stay out of the other sites' path.
template <int Q>
__device__ __noinline__ ElbmSite<Q> elbm_f32_far(const Params& p, ElbmSite<Q> in) {
    const float* f = in.F;
    ElbmSite<Q> o = in;
    o.code = -1;
    o.iters = 1;
    FfSite<Q> s;
    ff_site<Q, true>(f, s);
    float fmin = 1e30f, q = 0.f, amax = 0.f;
    bool neg = false;
    Ff d[Q], fe[Q], far = {0.f, 0.f};  // far: the largest -d
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        fe[i] = two_sum(s.Dh[i], f[i]);
        fe[i].l = fadd(fe[i].l, s.Dl[i]);
        d[i] = ff_div(fast_two_sum(s.Dh[i], s.Dl[i]), fe[i]);
        neg |= f[i] < 0.f;
        fmin = fminf(fmin, __fdividef(f[i], fe[i].h));
        q = fmaf(s.Dh[i], d[i].h, q);
        amax = fmaxf(amax, fabsf(d[i].h));
        if (-d[i].h > far.h) far = Ff{-d[i].h, -d[i].l};
    }
    // (Delta S >= q / (2 + 2 amax / 3): g(x) >= x^2 / (2 + 2 x / 3))
    const bool ok = s.rho >= kFfRhoMin && s.rho <= kFfRhoMax && fabsf(s.ux) <= kFfUMax && fabsf(s.uy) <= kFfUMax &&
                    amax <= 4.f && far.h > 0x1p-20f && (neg || fmin >= 0x1p-12f) &&
                    0.99f * q / (2.f + 0.67f * amax) > p.elbm_thr[0] + p.elbm_thr[1] * s.rho;
    if (!ok) return o;
    // a = alpha - 1 = 1 / max(-d): f stays >= 0 up to there
    const Ff hi0 = ff_div(Ff{1.f, 0.f}, far);
    float y = 0.f;
    bool fallback = neg;
    if (!neg) {
        Ff gm[Q];
        float sc = 0.f, ln;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            gm[i] = ff_g(Ff{-d[i].h, -d[i].l}, ln);
            sc = fmaf(fe[i].h, gm[i].h, sc);
        }
        // H(a) = sum f* (g(a d) - g(-d)) = -S_f, convex, H(0) < 0: Newton inside
        // a bracket on FP32 values, the last steps on double-single ones
        float a = 1.f < hi0.h ? 1.f : 0.5f * hi0.h, lo = 0.f, hi = hi0.h, step = 0.f;
        bool exists = false, fine = false, settled = false;
        for (int k = 0; k < 16 && !settled && !fallback; ++k) {
            float H = 0.f, dH = 0.f;
            if (!fine) {
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const float x = a * d[i].h, l = log1pf(x);
                    H = fmaf(fe[i].h, fmaf(1.f + x, l, -x) - gm[i].h, H);
                    dH = fmaf(fe[i].h * d[i].h, l, dH);
                }
            } else {
                Ff acc = {0.f, 0.f};
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const Ff x = ff_mul(Ff{a, 0.f}, d[i]), g = ff_g(fast_two_sum(x.h, x.l), ln);
                    Ff t = two_sum(g.h, -gm[i].h);
                    t = fast_two_sum(t.h, fadd(t.l, fsub(g.l, gm[i].l)));
                    t = ff_mul(fe[i], t);
                    const Ff u = two_sum(acc.h, t.h);
                    acc = Ff{u.h, fadd(acc.l, fadd(u.l, t.l))};
                    dH = fmaf(fe[i].h * d[i].h, ln, dH);
                }
                H = acc.h + acc.l;
            }
            step = __fdividef(H, dH);
            if (H < 0.f) {
                lo = a;
                if (!exists && !(dH > 0.f && a - step < 0.999f * hi0.h)) {
                    // does H reach zero below hi0?  Its sign at hi0, where it is
                    // clear of FP32 rounding, decides
                    float e = 0.f;
#pragma unroll
                    for (int i = 0; i < Q; ++i) {
                        const float x = hi0.h * d[i].h;
                        e = fmaf(fe[i].h, x <= -0.999999f ? 1.f : (1.f + x) * log1pf(x) - x, e);
                    }
                    if (!(fabsf(e - sc) > 1e-3f * sc)) return o;
                    fallback = e < sc;  // no root: the configured rule
                }
            } else {
                hi = a;
            }
            exists = true;
            const float next = a - step;
            const bool close = dH > 0.f && fabsf(step) <= 1e-4f * a && next < hi0.h;
            // what a last step leaves is H'' / (2 H') step^2.  A root next to
            // a = hi0 has one small 1 + x = w there, H'' / H' <= 1 / (a w |ln w|),
            // and w > 1.2e-4 (w (1 - ln w) > 1e-3 by the margin above): below
            // 450 step^2 / a, 0.44 x 2^-24 a for steps up to 2^-17 a (measured up
            // to there: 0.28 x 2^-24 of alpha)
            settled = fine && close && fabsf(step) <= 0x1p-17f * a;
            if (!settled) a = close || (dH > 0.f && next > lo && next < hi) ? next : 0.5f * (lo + hi);
            if (close && !fine) {  // FP32 rounding may have put a bound on the wrong side
                fine = true;
                lo = 0.f;
                hi = hi0.h;
            }
        }
        if (!settled && !fallback) return o;
        y = (a - 1.f) - step;
    }
    o.code = 0;
    if (fallback) {
        y = p.elbm_fallback == LBM_FALLBACK_EHRENFEST ? -1.f : (hi0.h - 1.f) + hi0.l;
        o.code = 2;
        o.iters = 0;
    }
    const float ab = p.beta2[0] + fmaf(y, p.beta_f, p.beta2[1]);
#pragma unroll
    for (int i = 0; i < Q; ++i) o.F[i] = fmaf(ab, s.Dh[i] + s.Dl[i], f[i]);
    conserve_mass<Q, float>(s.rho, o.F);
    return o;
}

// The FP64 solve for a site outside the range of the FP32 forms (a negative,
// vanishing or non-finite population, a large velocity or extreme density) or
// too close to the near-equilibrium threshold to settle in FP32.  Out of
// line, so that its registers and FP64 work stay out of the other sites'
// path.
template <int Q>
__device__ __noinline__ ElbmSite<Q> elbm_fp64_site(const Params& p, ElbmSite<Q> in) {
    double fd[Q], fe[Q], D[Q], r, a, b;
#pragma unroll
    for (int i = 0; i < Q; ++i) fd[i] = (double)in.F[i];
    moments<Q, double>(fd, r, a, b);
    equilibrium<Q, double>(LBM_EQ_ENTROPIC, r, a, b, fe);
#pragma unroll
    for (int i = 0; i < Q; ++i) D[i] = fe[i] - fd[i];
    const ElbmOut out = elbm_alpha<Q>(fd, fe, D, r, p);
    const float abf = (float)(out.alpha * p.beta);
    ElbmSite<Q> o;
#pragma unroll
    for (int i = 0; i < Q; ++i) o.F[i] = fmaf(abf, (float)D[i], in.F[i]);
    elbm_conserve<Q>(in.F, o.F);
    o.code = out.code;
    o.iters = out.iters;
    return o;
}

// The same for the few such sites of a warp (the lanes in `mask`), one group
// of lanes per site (elbm_lanes): a thread's own solve is a chain of about
// 1,000 FP64 operations of 64 clocks each.
template <int Q>
__device__ __noinline__ ElbmSite<Q> elbm_fp64_lanes(const Params& p, ElbmSite<Q> in, unsigned mask) {
    constexpr int G = ElbmLanes<Q>::G, S = 32 / G;
    const int lane = threadIdx.x & 31, g = lane / G, q = lane & (G - 1);
    ElbmSite<Q> o = in;
    while (mask) {
        // group k takes the k-th lane of the mask
        int src = -1, mine = -1;
#pragma unroll
        for (int k = 0; k < S; ++k) {
            const int l = mask ? __ffs(mask) - 1 : -1;
            if (k == g) src = l;
            if (l == lane) mine = k;
            mask &= mask - 1;  // 0 stays 0
        }
        float fq = 0.f;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const float v = __shfl_sync(0xffffffffu, in.F[i], src < 0 ? 0 : src);
            if (q == i) fq = v;
        }
        const ElbmLane e = elbm_lanes<Q>(p, (double)fq, src >= 0);
        const float Fq = fmaf((float)(e.alpha * p.beta), (float)e.D, fq);
        const int from = mine < 0 ? 0 : mine * G;
        const int code = __shfl_sync(0xffffffffu, e.code, from), it = __shfl_sync(0xffffffffu, e.iters, from);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const float v = __shfl_sync(0xffffffffu, Fq, from + i);
            if (mine >= 0) o.F[i] = v;
        }
        if (mine >= 0) {
            o.code = code;
            o.iters = it;
            elbm_conserve<Q>(in.F, o.F);
        }
    }
    return o;
}
// Sites of a warp up to which the groups of lanes take them: each round of
// 32 / G sites costs about a third of the threads' own solve.
template <int Q>
constexpr int kElbmLanesMost = Q == 9 ? 6 : 12;

// The ELBM collision F = f + alpha beta (f* - f) of one site in FP32; false
// where the site needs the FP64 solve.  e_code, e_iters: as ElbmOut's (a site
// solved here counts one step, the double-single one).
template <int Q>
__device__ __forceinline__ bool elbm_f32(const Params& p, const float* f, float* F, int& e_code, int& e_iters) {
    FfSite<Q> s;
    ff_site<Q, false>(f, s);
    if (!(s.rho > 0.f) || !(fabsf(s.ux) < 1e30f) || !(fabsf(s.uy) < 1e30f))
        if (*(volatile unsigned*)&p.counters[CNT_DIVERGED] == 0u) atomicExch(&p.counters[CNT_DIVERGED], 1u);
    // d = x, q = sum (f* - f)^2 / f*, amax = max |x|
    float q = 0.f, amax = 0.f, d[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const float D = s.Dh[i] + s.Dl[i];
        d[i] = __fdividef(D, s.Dh[i] + f[i]);
        q = fmaf(D, d[i], q);
        amax = fmaxf(amax, fabsf(d[i]));
    }
    // Delta S of the site lies in (q / 2) [1 - amax / 3, 1 + amax] (elbm_skip_certain's
    // series).  |x| is about 1e-7 at the threshold, where f* - f is good to
    // 2e-5 of itself (2^-40 f* at |u| = 0.4): the factors 1 +- 5e-5 cover q's error
    const float thr = p.elbm_thr[0] + p.elbm_thr[1] * s.rho;
    const bool in_range = s.rho >= kFfRhoMin && s.rho <= kFfRhoMax && amax < ff_x_limit(s.ux, s.uy);
    const bool skip = 0.5f * q * (1.f + amax) * 1.00005f < thr;
    const bool solve = 0.5f * q * (1.f - 0.34f * amax) * 0.99995f > thr;
    if (!in_range || !(skip || solve)) return false;
    float y = 0.f;
    e_code = skip ? 1 : 0;
    if (!skip) {
        e_iters = 1;
        if (amax < 0x1p-7f)
            y = f_root<Q>(s, d, q);
        else if (amax < 0x1p-4f)
            y = ff_root<Q, 10>(f, s);
        else
            y = ff_root<Q, 16>(f, s);
    }
    // alpha beta = 2 beta + y beta, 2 beta in two floats
    const float ab = p.beta2[0] + fmaf(y, p.beta_f, p.beta2[1]);
#pragma unroll
    for (int i = 0; i < Q; ++i) F[i] = fmaf(ab, s.Dh[i] + s.Dl[i], f[i]);
    conserve_mass<Q, float>(s.rho, F);
    return true;
}

// The collision for the sites of one warp (every lane calls it; valid: the
// lane has a site).
template <int Q>
__device__ __forceinline__ void elbm_warp(const Params& p, bool valid, const float* f, float* F, int& e_code,
                                          int& e_iters) {
    bool hard = valid && !elbm_f32<Q>(p, f, F, e_code, e_iters);
    if (!__any_sync(0xffffffffu, hard)) return;
    ElbmSite<Q> o;
#pragma unroll
    for (int i = 0; i < Q; ++i) o.F[i] = f[i];
    const bool was = hard;
    if (hard) {
        o = elbm_f32_far<Q>(p, o);
        hard = o.code < 0;
    }
    const unsigned mask = __ballot_sync(0xffffffffu, hard);
    if (mask) {
        if (__popc(mask) <= kElbmLanesMost<Q>)
            o = elbm_fp64_lanes<Q>(p, o, mask);
        else if (hard)
            o = elbm_fp64_site<Q>(p, o);
    }
    if (was) {
#pragma unroll
        for (int i = 0; i < Q; ++i) F[i] = o.F[i];
        e_code = o.code;
        e_iters = o.iters;
    }
}

}  // namespace lbm
