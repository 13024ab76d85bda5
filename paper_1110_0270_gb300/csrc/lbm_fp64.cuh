// D2Q9 collisions in FP64 storage with as few FP64-pipe instructions as the
// arithmetic needs.
//
// Why: a GB300 SM finishes one FP64 warp instruction (add, mul, fma, compare,
// conversion alike) in 19 clocks, so the FP64 step's time is its count of
// them: 2049^2 LBGK ran 6.3 GLUPS at 13% of the HBM rate, about 80 of them a
// site.  Here opposite
// populations share their sums and differences, f* - f is one fma per
// population (its product is not rounded before the subtraction), 1 / rho and
// the square roots are Newton steps from an FP32 seed, MRT works on the sums
// and differences of opposite pairs, and the divergence test, the signs and
// the limiter screen's FP32 copies are taken from the bits by integer
// instructions.
#pragma once

#include "lbm_device.cuh"

namespace lbm {

// v in FP32, truncated toward zero, by integer instructions; magnitudes below
// 2^-126 give 0 and above 2^127 (2 - 2^-23) that value (non-finite v too).
__device__ __forceinline__ float trunc_f32(double v) {
    const int hi = __double2hiint(v), lo = __double2loint(v);
    int e = (hi & 0x7fffffff) - 0x38000000;  // exponent rebased from 1023 to 127
    const bool tiny = e < 0x100000, huge = e >= 0x0ff00000;
    unsigned b = __funnelshift_l((unsigned)lo, (unsigned)e, 3);
    b = tiny ? 0u : (huge ? 0x7f7fffffu : b);
    return __uint_as_float(b | ((unsigned)hi & 0x80000000u));
}
// A normal positive float as a double.
__device__ __forceinline__ double widen_f64(float v) {
    const unsigned b = __float_as_uint(v);
    return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}
// hi words of 2^-100 and 2^100: the range in which the seeds below are normal.
__device__ __forceinline__ bool seedable(double a) {
    return (unsigned)(__double2hiint(a) - 0x39b00000) < 0x0c800000u;
}
// 1 / a: an FP32 seed (relative error e0 <= 2^-22) and one third-order step
// r (1 + e + e^2), whose own error is e0^3 = 2^-66.
__device__ __forceinline__ double rcp_f64(double a) {
    if (!seedable(a)) return 1.0 / a;
    float s;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(trunc_f32(a)));
    const double r = widen_f64(s), e = fma(-a, r, 1.0);
    return fma(r, fma(e, e, e), r);
}
// sqrt(a): an FP32 seed of 1 / sqrt(a) and two Newton steps of the root.
__device__ __forceinline__ double sqrt_f64(double a) {
    if (!seedable(a)) return sqrt(a);
    float s;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(trunc_f32(a)));
    const double h = widen_f64(0.5f * s);
    double r = a * widen_f64(s);
    r = fma(fma(-r, r, a), h, r);
    return fma(fma(-r, r, a), h, r);
}

// !(rho > 0) or a velocity of magnitude 1e30 or above (or NaN), by the bits.
__device__ __forceinline__ bool state_bad(double rho, double ux, double uy) {
    const int r = __double2hiint(rho);
    const unsigned x = __double2hiint(ux) & 0x7fffffff, y = __double2hiint(uy) & 0x7fffffff;
    constexpr unsigned big = 0x46293e59;  // hi word of 1e30
    const bool pos = r > 0 ? r <= 0x7ff00000 : (r == 0 && __double2loint(rho) != 0);
    return !pos || x >= big || y >= big;
}

// Moments and the factors of f*: f*_i = X[cx + 1] Y[cy + 1] (product
// equilibria; X carries rho), or the textbook polynomial's parts.
struct Eq64 {
    double rho, ux, uy, X[3], Y[3];
};

__device__ __forceinline__ void moments_f64(const double* f, Eq64& m) {
    // pairs (1, 5), (3, 7), (2, 6), (4, 8)
    const double a = f[1] + f[5], b = f[3] + f[7], c = f[2] + f[6], d = f[4] + f[8];
    const double p = f[1] - f[5], q = f[7] - f[3], r = f[2] - f[6], s = f[8] - f[4];
    m.rho = f[0] + ((a + b) + (c + d));
    const double jx = p + (r + s), jy = q + (s - r);
    const double inv = rcp_f64(m.rho);
    m.ux = jx * inv;
    m.uy = jy * inv;
    m.X[0] = jx;  // kept for factors_f64
}

// Product equilibria: 1D factors a -+ u / 2, 1 - 2a, a = 1/6 + u^2 / 2
// (polynomial) or (2 sqrt(1 + 3 u^2) - 1) / 6 (entropic); the x ones times rho.
__device__ __forceinline__ void factors_f64(int kind, Eq64& m) {
    const double hx = 0.5 * m.X[0], hy = 0.5 * m.uy;
    double A, a;
    if (kind == LBM_EQ_ENTROPIC) {
        A = m.rho * fma(sqrt_f64(fma(3.0 * m.ux, m.ux, 1.0)), 1.0 / 3.0, -1.0 / 6.0);
        a = fma(sqrt_f64(fma(3.0 * m.uy, m.uy, 1.0)), 1.0 / 3.0, -1.0 / 6.0);
    } else {
        A = fma(hx, m.ux, m.rho * (1.0 / 6.0));
        a = fma(hy, m.uy, 1.0 / 6.0);
    }
    m.X[0] = A - hx;
    m.X[1] = fma(-2.0, A, m.rho);
    m.X[2] = A + hx;
    m.Y[0] = a - hy;
    m.Y[1] = fma(-2.0, a, 1.0);
    m.Y[2] = a + hy;
}

// e_i = f*_i - f_i.
template <int FIRST>
__device__ __forceinline__ void diff_f64(int kind, const Eq64& m, const double* f, double* e) {
    using L = Lat<9>;
    if (kind == LBM_EQ_POLY_STD) {
        // textbook: f*_i = W_i rho (k + 3 cu + 4.5 cu^2), k = 1 - 1.5 u^2; the
        // rest population as rho minus the others
        const double k = fma(-1.5, fma(m.ux, m.ux, m.uy * m.uy), 1.0);
        const double ra = m.rho * (1.0 / 9.0), rd = m.rho * (1.0 / 36.0);
        const double s = m.ux + m.uy, t = m.ux - m.uy;
        double fe[9], rest = m.rho;
        // pairs (i, opp i) along x, y and the two diagonals
        const double cu[4] = {m.ux, m.uy, s, t};
        const int up[4] = {1, 7, 8, 2};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const double R = fma(4.5 * cu[j], cu[j], k), P = 3.0 * cu[j], w = j < 2 ? ra : rd;
            const int i = up[j], o = L::opp(i);
            fe[i] = w * (R + P);
            fe[o] = w * (R - P);
            e[i] = fma(w, R + P, -f[i]);
            e[o] = fma(w, R - P, -f[o]);
            if (FIRST == 0) rest -= fe[i] + fe[o];
        }
        if (FIRST == 0) e[0] = rest - f[0];
        return;
    }
#pragma unroll
    for (int i = FIRST; i < 9; ++i) e[i] = fma(m.X[L::cx(i) + 1], m.Y[L::cy(i) + 1], -f[i]);
}

// The limiter screen (maybe_above_loose's argument) on e = f* - f in FP32:
// s2 = sum e^2 and a lower bound of min f*; both inputs are truncated, which
// the 0.2% margin of the first test and the slack of the second cover.
__device__ __forceinline__ bool screen_f64(int kind, const Eq64& m, const double* f, const double* e, float delta) {
    float s2 = 0.f, mn;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const float v = trunc_f32(e[i]);
        s2 = fmaf(v, v, s2);
    }
    if (kind == LBM_EQ_POLY_STD) {
        mn = INFINITY;
#pragma unroll
        for (int i = 0; i < 9; ++i) mn = fminf(mn, trunc_f32(f[i] + e[i]));
    } else {
        const float x = fminf(fminf(trunc_f32(m.X[0]), trunc_f32(m.X[1])), trunc_f32(m.X[2]));
        const float y = fminf(fminf(trunc_f32(m.Y[0]), trunc_f32(m.Y[1])), trunc_f32(m.Y[2]));
        mn = fmaxf(x, 0.f) * fmaxf(y, 0.f);  // 0: never quiet
    }
    const float rho = trunc_f32(m.rho);
    if (mn > 0.f && s2 < mn * fminf(0.25f * mn, 0.998f * delta) && rho < 1e6f * delta) return false;
    if (!(mn > 0.f) || !(s2 < 0.25f * mn * mn)) return true;
    const float q = __fdividef(s2, mn);
    return slack_reaches(q, q, rho, delta);
}

// The collisions that run this form.
template <int Q, class T, int COLL>
constexpr bool kFp64Form = Q == 9 && sizeof(T) == 8 &&
                           (COLL == LBM_LBGK || COLL == LBM_EHRENFEST || COLL == LBM_POSITIVITY || COLL == LBM_MRT ||
                            COLL == LBM_MRT2 || COLL == LBM_MRT_LIMITER);

// LBGK: F_i = f_i + 2 beta e_i (i > 0; the rest population by mass).
__device__ __forceinline__ void lbgk_f64(double om, const double* f, const double* e, double* F) {
#pragma unroll
    for (int i = 1; i < 9; ++i) F[i] = fma(om, e[i], f[i]);
}

// A_2 (mrt2_d2q9): F = f* + (1 - s_nu)/4 (m4 r4 + m5 r5), m = r . (f - f*);
// c = (s_nu - 1) / 4.
__device__ __forceinline__ void mrt2_f64(double c, const double* f, const double* e, double* F) {
    const double m4 = c * ((e[1] + e[5]) - (e[3] + e[7])), m5 = c * ((e[4] + e[8]) - (e[2] + e[6]));
    F[1] = (f[1] + e[1]) + m4;
    F[5] = (f[5] + e[5]) + m4;
    F[3] = (f[3] + e[3]) - m4;
    F[7] = (f[7] + e[7]) - m4;
    F[4] = (f[4] + e[4]) + m5;
    F[8] = (f[8] + e[8]) + m5;
    F[2] = (f[2] + e[2]) - m5;
    F[6] = (f[6] + e[6]) - m5;
}

// MRT of Section 5 (mrt_d2q9) on the pair sums and differences of
// e = f* - f.  With sum e = 0 and sum v e = 0 the moments of M1 are
//   e: 3 (A + 2 D), eps: -3 (2 A + D), q_x: -3 (e_1 - e_5), q_y: 3 (e_3 - e_7),
//   p_xx: S_1 - S_3, p_xy: S_4 - S_2,
// A and D the sums over the axis and the diagonal populations, S_i the sum of
// the pair i.
__device__ __forceinline__ void mrt_f64(const Mrt64& r, const double* f, const double* e, double* F) {
    const double S1 = e[1] + e[5], S3 = e[3] + e[7], S2 = e[2] + e[6], S4 = e[4] + e[8];
    const double A = S1 + S3, D = S2 + S4;
    // even parts: axis rows -e - 2 eps, diagonal rows 2 e + eps
    const double ax = fma(r.aA, A, r.aD * D), dg = fma(r.dA, A, r.dD * D);
    const double pxx = r.nu * (S1 - S3), pxy = r.nu * (S4 - S2);
    const double a1 = ax + pxx, a3 = ax - pxx, d2 = dg - pxy, d4 = dg + pxy;
    const double dx = e[1] - e[5], dy = e[3] - e[7];
    // the q_x row with q_x = -q dx, the q_y row with q_y = q dy
    const double ox = r.q2 * dx, oy = r.q2 * dy;
    const double u = r.q * (dx + dy), v = r.q * (dx - dy);
    F[1] = f[1] + (a1 + ox);
    F[5] = f[5] + (a1 - ox);
    F[3] = f[3] + (a3 + oy);
    F[7] = f[7] + (a3 - oy);
    // 2 SE: q_x - q_y, 6 NW: its negative; 4 SW: -q_x - q_y, 8 NE: its negative
    F[2] = f[2] + (d2 - u);
    F[6] = f[6] + (d2 + u);
    F[4] = f[4] + (d4 + v);
    F[8] = f[8] + (d4 - v);
}

// The rest population as rho minus the others.
__device__ __forceinline__ void mass_f64(double rho, double* F) {
    F[0] = rho - (((F[1] + F[5]) + (F[3] + F[7])) + ((F[2] + F[6]) + (F[4] + F[8])));
}

// Delta S = sum f* g((f - f*) / f*) and q = sum (f - f*)^2 / f* of the state
// behind e = f* - f (delta_s_and_q's arithmetic): 1 / f* as the product of six
// reciprocals (nine divisions take 63 FP64 instructions), and one series
// length per site, from the exponent of the largest |x| (gfun_d picks one per
// population, with FP64 compares).  The first omitted term is below 2^-56 of
// the leading one in every tier.
template <int K>
__device__ __forceinline__ double gsum_f64(const double* x, const double* dx) {
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        double p = ((K & 1) ? -1.0 : 1.0) / (double)((K + 1) * (K + 2));
#pragma unroll
        for (int k = K - 1; k >= 0; --k) p = fma(p, x[i], ((k & 1) ? -1.0 : 1.0) / (double)((k + 1) * (k + 2)));
        s = i == 0 ? dx[0] * p : fma(dx[i], p, s);
    }
    return s;
}
__device__ __forceinline__ double delta_s_f64(int kind, const Eq64& m, const double* f, const double* e, double& q) {
    using L = Lat<9>;
    double x[9], dx[9];
    int top = 0, low = 0;  // hi words: the largest |x|; negative where an f* is not positive
    double rx[3], ry[3];
    if (kind != LBM_EQ_POLY_STD) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            rx[k] = -rcp_f64(m.X[k]);
            ry[k] = rcp_f64(m.Y[k]);
        }
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        // -1 / f*_i
        const double r = kind == LBM_EQ_POLY_STD ? -rcp_f64(f[i] + e[i]) : rx[L::cx(i) + 1] * ry[L::cy(i) + 1];
        low |= ~__double2hiint(r);  // r < 0 where f*_i > 0
        x[i] = e[i] * r;
        dx[i] = -(e[i] * x[i]);
        top = max(top, __double2hiint(x[i]) & 0x7fffffff);
    }
    q = ((dx[0] + (dx[1] + dx[5])) + (dx[3] + dx[7])) + ((dx[2] + dx[6]) + (dx[4] + dx[8]));
    if (low < 0) return __longlong_as_double(0x7ff0000000000000ULL);
    if (top < 0x3f300000) return gsum_f64<4>(x, dx);    // 2^-12
    if (top < 0x3f600000) return gsum_f64<5>(x, dx);    // 2^-9
    if (top < 0x3f900000) return gsum_f64<8>(x, dx);    // 2^-6
    if (top < 0x3fc00000) return gsum_f64<16>(x, dx);   // 1/8
    if (top < 0x3fd00000) return gsum_f64<26>(x, dx);   // 1/4
    double s = 0.0;
    bool neg = false;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        neg |= f[i] < 0.0;
        s += (f[i] + e[i]) * gfun_d(x[i]);
    }
    return neg ? __longlong_as_double(0x7ff0000000000000ULL) : s;
}

// x^k for x >= 0: the exponents the limiters use most without pow (about 150
// FP64 instructions); k is the same for every thread.
__device__ __forceinline__ double pow_f64(double x, double k) {
    const long long b = __double_as_longlong(k);
    if (b == 0x3ff0000000000000LL) return x;                // 1
    if (b == 0x3fe0000000000000LL) return sqrt(x);          // 1/2
    if (b == 0x4000000000000000LL) return x * x;            // 2
    if (b == 0x3ff8000000000000LL) return x * sqrt(x);      // 3/2
    if (b == 0LL) return 1.0;
    if (b == (long long)0xbfe0000000000000ULL) return 1.0 / sqrt(x);  // -1/2
    return pow(x, k);
}

}  // namespace lbm
