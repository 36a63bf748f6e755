// Integer-order Bessel functions J_l(x), Y_l(x), l = 0..nmax, x > 0, in FP64.
//
// Methods (all published; constants below are exact rationals or pi, gamma):
//  * x <= 20: J. C. P. Miller's backward recurrence (1952) from an order
//    well above max(nmax, x), normalised with J_0 + 2 sum_{j>=1} J_{2j} = 1.
//    The same sweep accumulates the Neumann series of Abramowitz & Stegun
//    9.1.88,
//        (pi/2) Y_0 = (ln(x/2) + gamma) J_0 - 2 sum_{k>=1} (-1)^k J_{2k} / k,
//    and its derivative (Y_1 = -Y_0', J_{2k}' = (J_{2k-1} - J_{2k+1})/2),
//        (pi/2) Y_1 = (ln(x/2) + gamma) J_1 - J_0 / x
//                     + sum_{k>=1} (-1)^k (J_{2k-1} - J_{2k+1}) / k.
//  * x > 20: Hankel's asymptotic expansion (A&S 9.2.5, 9.2.6, 9.2.9,
//    9.2.10) for J_0, J_1, Y_0, Y_1, its terms down to 2e-18 (the count is
//    taken from the size of x; at x > 20 the smallest term is below
//    e^{-40}); the phase x - (nu/2 + 1/4) pi is formed from sin x and cos x
//    so that no rounded multiple of pi is subtracted from a large x.  J_l for
//    l > 1 then comes from the forward recurrence when nmax <= x, else from
//    Miller's sweep.
//  * Y_l, l >= 2: forward recurrence Y_{l+1} = (2l/x) Y_l - Y_{l-1}
//    (Y is the dominant solution, so this direction is stable).
//
// The FP64 pipe (2 lanes per clock and SM: 64 clocks for a warp-wide
// instruction) bounds every caller, so no step divides: 2l/x is 2l times the
// reciprocal of x kept as a sum of two doubles (TwoOverX, as accurate as the
// quotient), 1/k comes from a table and Hankel's coefficients are constants.
#pragma once

#include <math.h>

#define MSD_EULER_GAMMA 0.57721566490153286061

// Start order of the backward recurrence: past the turning point by a
// margin growing like sqrt(order), so that J_start / J_nmax is far below
// the FP64 unit roundoff.
__host__ __device__ __forceinline__ int miller_start(int nmax, double x) {
    double top = fmax((double)nmax, x);
    int s = (int)(top + sqrt(60.0 * top)) + 16;
    return s + (s & 1);  // even
}

// 2l/x for integer l without a division: 2/x = hi + lo to about 100 bits.
struct TwoOverX {
    double hi, lo;
    __device__ explicit TwoOverX(double x) {
        hi = 2.0 / x;
        lo = fma(-x, hi, 2.0) * (0.5 * hi);
    }
    __device__ double times(double l) const { return fma(l, hi, l * lo); }
};

// 1/k and 1/k + 1/(k+1) for the Neumann sums (k < 128 covers the start order
// of every nmax <= 2 MSD_MAX_N + 1), and the coefficients of Hankel's
// expansion: term k of order nu is c[nu][k] / x^k,
// c_k = c_{k-1} (4 nu^2 - (2k-1)^2) / (8k), with the signs of P and Q.
struct BesselTables {
    double recip[128], recip2[128];
    double hankel[2][32];
};
constexpr BesselTables make_bessel_tables() {
    BesselTables t{};
    for (int k = 1; k < 128; ++k) {
        t.recip[k] = 1.0 / k;
        t.recip2[k] = 1.0 / (k + 1) + 1.0 / k;
    }
    for (int nu = 0; nu < 2; ++nu) {
        double c = 1.0;
        t.hankel[nu][0] = 1.0;
        for (int k = 1; k < 32; ++k) {
            c *= (4.0 * nu * nu - (2.0 * k - 1.0) * (2.0 * k - 1.0)) / (8.0 * k);
            t.hankel[nu][k] = ((k >> 1) & 1) ? -c : c;
        }
    }
    return t;
}
static __constant__ BesselTables c_bessel = make_bessel_tables();

// Miller sweep: J[0..nmax] normalised; s0, s1 = the two Neumann sums above
// (already divided by the normalisation; SUMS false: not formed).
template <bool SUMS>
__device__ inline void bessel_miller(double x, int nmax, double* J, double* s0, double* s1) {
    const int start = miller_start(nmax, x);
    const TwoOverX f(x);
    const double small = 1e-250;
    double jp1 = 0.0, jl = 1e-30, norm = 0.0, a0 = 0.0, a1 = 0.0;
    // orders l (odd) and l - 1 (even) per round; start is even, so its own
    // (even) term opens the sums
    auto step = [&](int l) {
        if (l <= nmax) J[l] = jl;
        const double jm1 = fma(f.times((double)l), jl, -jp1);
        jp1 = jl;
        jl = jm1;
        // |jl| > 1e250 (by its exponent: 1023 + 830)
        if (((__double2hiint(jl) >> 20) & 0x7ff) > 1853) {
            jl *= small;
            jp1 *= small;
            norm *= small;
            a0 *= small;
            a1 *= small;
            for (int i = l; i <= nmax; ++i) J[i] *= small;
        }
    };
    for (int l = start; l >= 2; l -= 2) {
        const int k = l >> 1;  // l = 2k
        norm += jl;
        if (SUMS) a0 = fma((k & 1) ? -jl : jl, c_bessel.recip[k], a0);
        step(l);
        // l - 1 = 2(k-1) + 1: coefficient of J_{2k-1} in sum_k (-1)^k (J_{2k-1} - J_{2k+1}) / k
        if (SUMS) {
            if (k == 1) a1 -= jl;
            else a1 = fma((k & 1) ? -jl : jl, c_bessel.recip2[k - 1], a1);
        }
        step(l - 1);
    }
    J[0] = jl;
    const double inv = 1.0 / fma(2.0, norm, jl);  // J_0 + 2 sum J_2k
    for (int i = 0; i <= nmax; ++i) J[i] *= inv;
    if (SUMS) {
        *s0 = a0 * inv;
        *s1 = a1 * inv;
    }
}

// Hankel's expansion of orders 0 and 1, x > 20, given sin x and cos x.
__device__ inline void bessel_asymptotic01(double x, double sx, double cx, double* J0, double* Y0, double* J1,
                                           double* Y1) {
    // terms k < K (K even: K / 2 of P and of Q) down to 2e-18
    const int K = x < 25.0 ? 32 : x < 40.0 ? 22 : x < 100.0 ? 16 : x < 300.0 ? 10 : 8;
    const double u = 1.0 / x, v = u * u;
    double P0 = 0.0, Q0 = 0.0, P1 = 0.0, Q1 = 0.0;
    for (int k = K - 2; k >= 0; k -= 2) {
        P0 = fma(P0, v, c_bessel.hankel[0][k]);
        Q0 = fma(Q0, v, c_bessel.hankel[0][k + 1]);
        P1 = fma(P1, v, c_bessel.hankel[1][k]);
        Q1 = fma(Q1, v, c_bessel.hankel[1][k + 1]);
    }
    Q0 *= u;
    Q1 *= u;
    // sqrt(2/(pi x)) times cos and sin of x - (nu/2 + 1/4) pi, the 1/sqrt(2) taken into the amplitude
    const double amp = sqrt(u * (1.0 / M_PI));
    const double p = (cx + sx) * amp, m = (sx - cx) * amp;
    *J0 = P0 * p - Q0 * m;
    *Y0 = P0 * m + Q0 * p;
    *J1 = P1 * m + Q1 * p;
    *Y1 = Q1 * m - P1 * p;
}

// J[0..nmax], Y[0..nmax] (caller arrays of length >= max(nmax, 1) + 1).
__device__ inline void bessel_jy(double x, int nmax, double* J, double* Y) {
    const int nm = nmax < 1 ? 1 : nmax;
    const TwoOverX f(x);
    double Y0, Y1;
    if (x > 20.0) {
        double sx, cx;
        sincos(x, &sx, &cx);
        double J0, J1;
        bessel_asymptotic01(x, sx, cx, &J0, &Y0, &J1, &Y1);
        if ((double)nm <= x) {
            J[0] = J0;
            J[1] = J1;
            for (int l = 1; l < nm; ++l) J[l + 1] = fma(f.times((double)l), J[l], -J[l - 1]);
        } else {
            bessel_miller<false>(x, nm, J, nullptr, nullptr);
        }
    } else {
        double s0, s1;
        bessel_miller<true>(x, nm, J, &s0, &s1);
        const double L = log(0.5 * x) + MSD_EULER_GAMMA;
        Y0 = (2.0 / M_PI) * (L * J[0] - 2.0 * s0);
        Y1 = (2.0 / M_PI) * (L * J[1] - J[0] / x + s1);
    }
    Y[0] = Y0;
    Y[1] = Y1;
    for (int l = 1; l < nm; ++l) Y[l + 1] = fma(f.times((double)l), Y[l], -Y[l - 1]);
}
