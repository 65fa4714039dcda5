// Hankel functions of order 0 and 1 on the device, FP64: bessel_miller's recurrence and Neumann series
// (bessel.cuh) with the quotients of the series in tables.  FP64 instructions issue at one per
// 64 clocks here and a division is some twenty of them, so the two divisions a step were
// most of its work.  Same accuracy as bessel_miller (largest error, relative to the modulus, against long
// double for x = 0.1 .. 600: 5.1e-16 .. 5.5e-14, equal for both).
#pragma once

#include "bessel.cuh"

constexpr int HK_SERIES = 15, HK_NEUMANN = 256;
constexpr double HK_SERIES_MAX = 2.0;
struct HankelSeries {                        // of J_1 and Y_1 (DLMF 10.2.2, 10.8.1)
    double a[HK_SERIES], b[HK_SERIES];       // (-1)^k / (k! (k+1)!), times H_k + H_{k+1}
    constexpr HankelSeries() : a{}, b{} {
        double f = 1.0, h = 0.0;
        for (int k = 0; k < HK_SERIES; ++k) {
            if (k > 0) { f /= -(double)k * (k + 1); h += 1.0 / k; }
            a[k] = f;
            b[k] = f * (h + h + 1.0 / (k + 1));
        }
    }
};
struct HankelNeumann {                       // factor of J_{2i} in Y_0's sum and of J_{2i+1} in Y_1's
    double e[HK_NEUMANN], o[HK_NEUMANN];
    static constexpr double even(int i) { return i == 0 ? 0.0 : ((i & 1) ? -1.0 : 1.0) / i; }
    static constexpr double odd(int i) { return i == 0 ? -1.0 : ((i & 1) ? 1.0 : -1.0) * (1.0 / i + 1.0 / (i + 1)); }
    constexpr HankelNeumann() : e{}, o{} {
        for (int i = 0; i < HK_NEUMANN; ++i) { e[i] = even(i); o[i] = odd(i); }
    }
};
static __constant__ HankelSeries c_hk_series = HankelSeries();
static __device__ const HankelNeumann g_hk_neumann = HankelNeumann();

// H_1 (and with H0 also H_0) for x > 0 by the recurrence.
template <bool H0>
__device__ inline void hankel_recurrence(double x, cd* h0, cd* h1) {
    const int m = miller_start(x, 1);
    const double inv = 2.0 / x;
    double tp = 0.0, t = 1e-30, norm = 0.0, sy0 = 0.0, sy1 = 0.0, jd = m;
    for (int i = m / 2 - 1; i >= 0; --i) {                 // t = t_{2i+2} -> t_{2i+1} -> t_{2i}
        const bool in = i + 1 < HK_NEUMANN;
        norm += t;
        if (H0) {
            const double w = in ? __ldg(g_hk_neumann.e + i + 1) : (((i + 1) & 1) ? -1.0 : 1.0) / (i + 1);
            sy0 = fma(w, t, sy0);
        }
        tp = fma(jd * inv, t, -tp);
        const double w = in ? __ldg(g_hk_neumann.o + i) : ((i & 1) ? 1.0 : -1.0) * (1.0 / i + 1.0 / (i + 1));
        sy1 = fma(w, tp, sy1);
        t = fma((jd - 1.0) * inv, tp, -t);
        jd -= 2.0;
        if ((__double2hiint(t) & 0x7fffffff) > 0x73000000) {   // about 1e247
            t *= 1e-250; tp *= 1e-250; norm *= 1e-250; sy0 *= 1e-250; sy1 *= 1e-250;
        }
    }
    const double lg = log(0.5 * x) + HFMM_EULER_GAMMA;
    const double s = 1.0 / (2.0 * norm + t), j0 = t * s, j1 = tp * s;
    if (H0) *h0 = cmk(j0, HFMM_2_OVER_PI * (lg * j0 - 2.0 * sy0 * s));
    *h1 = cmk(j1, HFMM_2_OVER_PI * (lg * j1 - j0 / x + sy1 * s));
}

// H_1^(1)(x), x > 0; up to x = 2 the ascending series (its terms fall from the first on).
__device__ inline cd hankel1(double x) {
    if (x <= HK_SERIES_MAX) {
        const double q = 0.25 * x * x;
        double j = c_hk_series.a[HK_SERIES - 1], y = c_hk_series.b[HK_SERIES - 1];
#pragma unroll
        for (int k = HK_SERIES - 2; k >= 0; --k) {
            j = fma(j, q, c_hk_series.a[k]);
            y = fma(y, q, c_hk_series.b[k]);
        }
        j *= 0.5 * x;
        return cmk(j, HFMM_2_OVER_PI * ((log(0.5 * x) + HFMM_EULER_GAMMA) * j - 1.0 / x - 0.25 * x * y));
    }
    cd h1;
    hankel_recurrence<false>(x, nullptr, &h1);
    return h1;
}
