// The FP64 ELBM solve of one site by a group of lanes, one population per
// lane (4 lanes per D1Q3 site, 16 per D2Q9 site).
//
// Why: an FP64 warp instruction costs 64 clocks of latency and 19 clocks of
// its SM however few lanes are active (measured), so a lattice with fewer
// warps than SM sub-partitions is bound by the length of one site's chain of
// FP64 operations, which runs through all Q populations when a thread owns a
// site (about 1,000 operations).  Here the populations' series, logarithms
// and divisions run side by side, and only their sums cross lanes.
#pragma once

#include "lbm_fp64.cuh"

namespace lbm {

template <int Q>
struct ElbmLanes {
    static constexpr int G = Q == 9 ? 16 : 4;  // lanes per site
};

// Sum over the lanes of a group, in every lane.
template <int G, class T>
__device__ __forceinline__ T group_sum(T v) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
template <int G>
__device__ __forceinline__ float group_max(float v) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float warp_max(float v) {  // v >= 0
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}

// sum_k c[k] z^k, K coefficients by pairs (Estrin): a chain of log2 K steps
// instead of K.  c is overwritten.
template <int K>
__device__ __forceinline__ double estrin(double* c, double z) {
#pragma unroll
    for (int n = K; n > 1; n = (n + 1) / 2) {
#pragma unroll
        for (int k = 0; k < n / 2; ++k) c[k] = fma(c[2 * k + 1], z, c[2 * k]);
        if (n & 1) c[n / 2] = c[n - 1];
        z *= z;
    }
    return c[0];
}
// gl_series<KG, KL> with its series by pairs.
template <int KG, int KL>
__device__ __forceinline__ void gl_pairs(double x, double& g, double& l) {
    constexpr int K = KL > KG + 1 ? KL : KG + 1;
    double c[K];
#pragma unroll
    for (int j = 0; j < K; ++j) c[j] = ((j & 1) ? 1.0 : -1.0) / (double)(j + 2);
    const double m = x * estrin<K>(c, x);
    l = fma(x, m, x);
    g = x * fma(m, 1.0 + x, x);
}
// g(x) and ln(1 + x) by the area tangent series: with s = x / (2 + x),
// ln(1 + x) = 2 artanh s = 2 s (1 + s^2 R), R = sum_{k<K} s^2k / (2k + 3), and
// from x = 2 s / (1 - s), g(x) = x s (1 + s R (1 + s)): no cancellation in
// either.  Converges like (x / 2)^2k where the Taylor series has x^k: 9 terms
// for |x| < 1/4 (27), 17 for 1/2.  The first omitted term is below 2^-56 of
// the leading one.  |x| <= 1/2 (2 + x: no range check on its reciprocal).
template <int K>
__device__ __forceinline__ void gl_artanh(double x, double& g, double& l) {
    float seed;
    const double y = 2.0 + x;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(seed) : "f"(trunc_f32(y)));
    const double r = widen_f64(seed), e = fma(-y, r, 1.0);
    const double s = x * fma(r, fma(e, e, e), r);  // x / (2 + x), as in rcp_f64
    double c[K];
#pragma unroll
    for (int k = 0; k < K; ++k) c[k] = 1.0 / (double)(2 * k + 3);
    const double w = s * estrin<K>(c, s * s), s2 = s + s;
    l = fma(s2 * s, w, s2);
    g = (x * s) * fma(w, 1.0 + s, 1.0);
}

// g(x) and ln(1 + x) at one population; am >= |x| over the warp picks the
// series length, so that the lanes take one branch.  The sites next to a
// shock (|x| to 1/2) set the step's time, since it lasts as long as its
// longest chain: a Horner chain of 27 terms and log1p there made the 800-site
// tube 20.6 us a step, these series 14.4 (13.9 with two steps a launch).
__device__ __forceinline__ void gl_lane(double x, float am, double& g, double& l) {
    if (am < 0x1p-20f)
        gl_series<2, 2>(x, g, l);
    else if (am < 0x1p-10f)
        gl_pairs<5, 5>(x, g, l);
    else if (am < 0.015625f)
        gl_pairs<8, 9>(x, g, l);
    else if (am < 0.125f)
        gl_artanh<7>(x, g, l);
    else if (am < 0.25f)
        gl_artanh<9>(x, g, l);
    else if (am < 0.5f)
        gl_artanh<17>(x, g, l);
    else {
        const double xc = x < -1.0 ? -1.0 : x;
        l = log1p(xc);
        g = xc <= -1.0 ? 1.0 : (1.0 + xc) * l - xc;
        if (fabs(x) < 0.25) {  // the closed form cancels for the small ones
            double gs, ls;
            gl_artanh<9>(x, gs, ls);
            g = gs;
        }
    }
}
// The FP32 stage's g and ln(1 + x), by the same series: six terms to |x| = 1/2.
__device__ __forceinline__ void gl_lane_f(float x, float am, float& g, float& l) {
    if (am < 0.5f) {
        const float s = __fdividef(x, 2.f + x), z = s * s;
        float r = 1.f / 13.f;
#pragma unroll
        for (int k = 11; k >= 3; k -= 2) r = fmaf(r, z, 1.f / (float)k);
        const float w = s * r, s2 = s + s;
        l = fmaf(s2 * s, w, s2);
        g = (x * s) * fmaf(w, 1.f + s, 1.f);
    } else {
        const float xc = x < -1.f ? -1.f : x;
        l = log1pf(xc);
        g = fabsf(x) < 0.25f ? x * x * gpoly_f<11>(x) : (xc <= -1.f ? 1.f : (1.f + xc) * l - xc);
    }
}

// What a group found: alpha, how (ElbmOut's code), the FP64 steps, and this
// lane's f* - f; rho, u of the site.
struct ElbmLane {
    double alpha, D, rho, ux, uy;
    int code, iters;
};

// elbm_alpha (the same tests and iteration) on groups of lanes: lane q < Q of
// a group holds population q of its site in f.  Every lane of the warp calls
// it; a group without a site passes valid = false.
template <int Q>
__device__ ElbmLane elbm_lanes(const Params& p, double f, bool valid) {
    constexpr int G = ElbmLanes<Q>::G;
    const int lane = threadIdx.x & 31;  // callers use warps of consecutive threadIdx.x
    const int q = lane & (G - 1);
    const bool act = valid && q < Q;
    const int cx = Q == 3 ? q - 1 : ((q == 1 || q == 2 || q == 8) ? 1 : ((q == 4 || q == 5 || q == 6) ? -1 : 0));
    const int cy = Q == 3 ? 0 : ((q == 6 || q == 7 || q == 8) ? 1 : ((q == 2 || q == 3 || q == 4) ? -1 : 0));
    if (!act) f = 0.0;
    ElbmLane o;
    o.iters = 0;
    const double r = group_sum<G>(f);
    const double jx = group_sum<G>(cx > 0 ? f : (cx < 0 ? -f : 0.0));
    const double jy = Q == 9 ? group_sum<G>(cy > 0 ? f : (cy < 0 ? -f : 0.0)) : 0.0;
    const double ri = rcp_f64(valid ? r : 1.0);
    const double ux = jx * ri, uy = jy * ri;
    o.rho = r;
    o.ux = ux;
    o.uy = uy;
    // 1D factors: the lower half of a D2Q9 group works on x, the upper on y
    double u = Q == 9 && (q & 8) ? uy : ux;
    const double a = fma(sqrt_f64(fma(3.0 * u, u, 1.0)), 1.0 / 3.0, -1.0 / 6.0);
    const int base = lane & ~(G - 1);
    const double aX = Q == 9 ? __shfl_sync(0xffffffffu, a, base) : a;
    const double fX = cx == 0 ? 1.0 - 2.0 * aX : aX + (0.5 * cx) * ux;
    double fe = r * fX;
    if (Q == 9) {
        const double aY = __shfl_sync(0xffffffffu, a, base + 8);
        fe *= cy == 0 ? 1.0 - 2.0 * aY : aY + (0.5 * cy) * uy;
    }
    const double D = act ? fe - f : 0.0;
    const double d = act ? D * rcp_f64(fe) : 0.0;
    o.D = D;
    const float Df = (float)D, df = (float)d, fef = (float)fe, ff = (float)f;
    const float dmax = group_max<G>(fabsf(df));
    double gm, lm;
    gl_lane(-d, warp_max(fminf(fabsf(df), 2.f)), gm, lm);
    if (!act) gm = 0.0;
    const double dS = group_sum<G>(act ? fe * gm : 0.0);
    const unsigned gbits = (G == 16 ? 0xffffu : 0xfu) << base;
    const bool neg = (__ballot_sync(0xffffffffu, act && f < 0.0) & gbits) != 0u;
    // alpha_max = 1 + 1 / max(-d): the largest -d by its bits (a positive
    // double orders like its bit pattern)
    long long mb = act && d < 0.0 ? __double_as_longlong(-d) : 0ll;
#pragma unroll
    for (int s = G / 2; s > 0; s >>= 1) {
        const long long t = __shfl_xor_sync(0xffffffffu, mb, s);
        mb = t > mb ? t : mb;
    }
    const double rneg = __longlong_as_double(mb);
    const double amax = mb ? 1.0 + rcp_f64(rneg) : __longlong_as_double(0x7ff0000000000000ULL);
    const double fb = p.elbm_fallback == LBM_FALLBACK_EHRENFEST ? 1.0 : amax;
    o.code = 0;
    o.alpha = 2.0;
    bool done = !valid;
    if (!done && !neg && dS < 1e-15 + p.elbm_skip_rel * r) {
        o.code = 1;
        done = true;
    } else if (!done && neg) {
        o.alpha = fb;
        o.code = 2;
        done = true;
    }
    if (__all_sync(0xffffffffu, done)) return o;
    // the square of the norm of f* - f: the stopping test compares squares
    double nrm2 = group_sum<G>(p.elbm_norm == LBM_NORM_L1 ? fabs(D) : D * d);
    if (p.elbm_norm == LBM_NORM_L1) nrm2 *= nrm2;
    const double eps2 = p.elbm_eps * p.elbm_eps;
    double al = 2.0 < amax ? 2.0 : 0.5 * (1.0 + amax);
    {
        // FP32 parabola iterations (elbm_alpha's): each cubes the error, so a
        // move of 1/500 leaves less than FP32 resolves, and the FP64 steps
        // that follow are of the same order.  Approximate divisions and root:
        // only the starting point depends on them.  (With log1pf, divisions and
        // a stop at 1e-6 this stage was a third of the warp's 2,800 instructions.)
        const float gmf = (float)gm, amf = (float)amax;
        float af = (float)al, lof = 1.f, hif = amf;
        bool fin = done;
        for (int k = 0; k < 8 && !__all_sync(0xffffffffu, fin); ++k) {
            const float x = (af - 1.f) * df;
            float g, l;
            gl_lane_f(x, warp_max(fin ? 0.f : fabsf(x)), g, l);
            const float t0 = group_sum<G>(act ? fef * (gmf - g) : 0.f);
            const float t1 = group_sum<G>(act ? -Df * l : 0.f);
            const float t2 = group_sum<G>(act ? -__fdividef(Df * Df, fmaxf(ff + af * Df, 1e-37f)) : 0.f);
            if (t0 > 0.f)
                lof = fin ? lof : af;
            else
                hif = fin ? hif : af;
            const float disc = t1 * t1 - 2.f * t0 * t2;
            float next = __int_as_float(0x7fc00000);
            if (disc >= 0.f) {
                float root;
                asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(root) : "f"(disc));
                const float w = -0.5f * (t1 + copysignf(root, t1));
                next = af + fmaxf(__fdividef(w, 0.5f * t2), __fdividef(t0, w));
            }
            if (!(next > lof && next < hif)) next = 0.5f * (lof + hif);
            const bool last = fabsf(next - af) <= 2e-3f * af;
            if (!fin) af = next;
            fin = fin || last;
        }
        const double ad = (double)af;
        if (ad > 1.0 && ad < amax) al = ad;
    }
    double s0, s1, lo = 1.0, hi = amax;
    float s2;
    auto eval = [&](double at, bool on) {
        const double x = on ? (at - 1.0) * d : 0.0;
        double g, l;
        gl_lane(x, warp_max(on ? fminf(fabsf((float)at - 1.f) * dmax, 2.f) : 0.f), g, l);
        const double t0 = group_sum<G>(act ? fe * (gm - g) : 0.0), t1 = group_sum<G>(act ? -D * l : 0.0);
        const float t2 = group_sum<G>(act ? -__fdividef(Df * Df, fmaxf(ff + (float)at * Df, 1e-37f)) : 0.f);
        if (on) {
            s0 = t0;
            s1 = t1;
            s2 = t2;
        }
    };
    s0 = s1 = 0.0;
    s2 = 0.f;
    eval(al, !done);
    {
        // no tangent zero below alpha_max: S_f(alpha_max) decides existence
        const bool look = !done && s0 > 0.0 && !(s1 < 0.0 && s0 < (al - amax) * s1);
        if (__any_sync(0xffffffffu, look)) {
            const double k0 = s0, k1 = s1;
            const float k2 = s2;
            eval(amax, look);
            if (look && s0 > 0.0) {
                o.alpha = fb;
                o.code = 2;
                done = true;
            }
            s0 = k0;
            s1 = k1;
            s2 = k2;
        }
    }
    if (s0 > 0.0)
        lo = al;
    else
        hi = al;
    bool run = !done;
    while (true) {
        if (run && (o.iters >= p.elbm_max_iter || (s0 * s0) * nrm2 < eps2 * (s1 * s1))) run = false;
        if (__all_sync(0xffffffffu, !run)) break;
        // the greater root of the parabola: where S_f falls (s1 < 0) it is
        // t 2 / (1 + sqrt(1 - e)) with t = -s0 / s1, e = 2 s0 s2 / s1^2: t and
        // a correction that FP32 holds to 1e-7 of itself
        const double t = s0 * rcp_f64(-s1);
        const float e = -2.f * (float)t * s2 / (float)s1;
        const float w = 1.f + sqrtf(1.f - e);
        double next = fma(t, (double)__fdividef(e, w * w), al + t);
        if (!(s1 < 0.0) && run) {
            const double disc = s1 * s1 - 2.0 * s0 * (double)s2;
            next = __longlong_as_double(0x7ff8000000000000ULL);
            if (disc >= 0.0) {
                const double v = -0.5 * (s1 + copysign(sqrt(disc), s1));
                next = al + fmax(v / (0.5 * (double)s2), s0 / v);
            }
        }
        if (!(next > lo && next < hi)) next = 0.5 * (lo + hi);
        if (run) {
            ++o.iters;
            al = next;
        }
        eval(al, run);
        if (run) {
            if (s0 > 0.0)
                lo = al;
            else
                hi = al;
        }
    }
    if (!done) o.alpha = s0 < 0.0 ? fma(2.0 * s0, rcp_f64(-s1), al) : al;
    return o;
}

}  // namespace lbm
