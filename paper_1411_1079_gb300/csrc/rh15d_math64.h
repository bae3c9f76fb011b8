// rh15d_math64.h -- FP64 exponential, reciprocal, Voigt and dispersion
// functions of the FP64 paths, table-driven.
//
// GB300 issues FP64 at 1/64 of the FP32 rate, so the FP64 kernels are bound
// by the number of FP64 instructions and nothing else; these functions spend
// table reads and integer work instead of FP64 operations.
//   exp: Tang (1989), table of 2^{j/64} and a degree-5 polynomial: 11 FP64
//     operations.
//   1/x: the hardware's approximation and two Newton steps: 4.
//   Voigt H(a, v) and dispersion L(a, v), w = H + i L, a <= 0.05: with F
//     Dawson's integral, w(z) = e^{-z^2} + (2i/sqrt pi) F(z), so that
//       H = e^{a^2 - v^2} cos 2av - (2/sqrt pi) [a F' - a^3/6 F''' + a^5/120 F^(5) - ...],
//       L = -e^{a^2 - v^2} sin 2av + (2/sqrt pi) [F - a^2/2 F'' + a^4/24 F^(4) - ...],
//     F and F' for |v| < 16 from their Taylor polynomials (degree 11) about
//     the centres of 128 intervals (both tabulated: F' = 1 - 2vF cancels),
//     the higher derivatives from F^(n+1) = -2 (v F^(n) + n F^(n-1)); for
//     |v| >= 16 the asymptotic series of w with as many terms as |v| needs
//     (6 to 10; the lanes of a warp reach from a line's core into its wings
//     and run both branches, so the branch point is where the second is short).  About 85 FP64 operations against some thousands of the
//     Dawson power series (one division a term, up to 130 terms), error
//     below 2e-15 relative where the series has up to 1e-14 (F' cancels
//     there).
#pragma once
#include <cmath>
#include <vector>

#include <cuda_runtime.h>

namespace rh {

constexpr int kV64N = 128;           // intervals of the Dawson tables
constexpr double kV64Max = 16.0;     // their range in |v|
constexpr int kV64Deg = 12;          // coefficients per polynomial
constexpr int kV64Row = 25;          // doubles per interval: F then F' (odd: spreads shared-memory banks)
constexpr int kT64Exp = kV64N * kV64Row;        // offset of 2^{j/64}
constexpr int kT64Dfac = kT64Exp + 64;          // offset of (2k-1)!!
constexpr int kT64Size = kT64Dfac + 18;         // doubles of the whole table

// The table, in long double on the host (rounded once; computed once per
// process: long double is emulated on some hosts, 3 ms).
inline std::vector<double> math64_table_build()
{
    std::vector<double> t(kT64Size, 0.0);
    for (int j = 0; j < kV64N; ++j) {
        const long double c = (2.0L * j + 1.0L) * (long double)kV64Max / (2.0L * kV64N);
        // F(c) = e^{-c^2} sum c^{2n+1} / (n! (2n+1))
        long double s = 0.0L, term = c;
        for (int n = 0; n < 400; ++n) {
            const long double q = term / (2 * n + 1);
            s += q;
            if (q < 1e-22L * s) break;
            term *= c * c / (n + 1);
        }
        long double a[kV64Deg + 2];
        a[0] = expl(-c * c) * s;
        a[1] = 1.0L - 2.0L * c * a[0];   // F', through its asymptotic form where this cancels
        if (c > 5.0L) {
            long double u = 1.0L / (2.0L * c * c), p = 1.0L, sum = 0.0L, last = 1e30L;
            for (int k = 1; k < 60; ++k) {
                p *= (2 * k - 1) * u;
                if (p > last) break;
                last = p;
                sum += p;
            }
            // used only where the series' smallest term is below the cancellation
            if (last < 1e-18L * sum) a[1] = -sum;
        }
        for (int k = 1; k <= kV64Deg; ++k) a[k + 1] = -2.0L * (c * a[k] + a[k - 1]) / (k + 1);
        for (int k = 0; k < kV64Deg; ++k) {
            t[j * kV64Row + k] = (double)a[k];
            t[j * kV64Row + kV64Deg + k] = (double)((k + 1) * a[k + 1]);
        }
    }
    for (int j = 0; j < 64; ++j) t[kT64Exp + j] = (double)exp2l(j / 64.0L);
    double f = 1.0;
    for (int k = 0; k < 18; ++k) {
        t[kT64Dfac + k] = f;   // (2k-1)!!
        f *= 2 * k + 1;
    }
    return t;
}

inline const std::vector<double> &math64_table()
{
    static const std::vector<double> t = math64_table_build();
    return t;
}

#ifdef __CUDACC__
// e^x; 0 below -708 (the true value is under 4e-308), for x <= 709
__device__ __forceinline__ double exp64(double x, const double *__restrict__ tab)
{
    const double magic = 6755399441055744.0;   // 1.5 * 2^52: rounds to an integer in the low word
    const double t = fma(x, 92.332482616893656877, magic);   // 64 / ln 2
    const int n = __double2loint(t);
    const double nd = t - magic;
    // ln 2 / 64 in two parts; nd * hi is exact
    double r = fma(nd, -0.0108304246959960437379777431488037109375, x);
    r = fma(nd, -2.5310172166650874898e-13, r);
    const double r2 = r * r;
    double p = fma(r, 1.0 / 120.0, 1.0 / 24.0);
    p = fma(r, p, 1.0 / 6.0);
    p = fma(r, p, 0.5);
    p = fma(r2, p, r);
    const double T = tab[kT64Exp + (n & 63)];
    const double v = fma(T, p, T);
    const double s = __hiloint2double(__double2hiint(v) + ((n >> 6) << 20), __double2loint(v));
    return x > -708.0 ? s : (x != x ? x : 0.0);
}

// 1/x for normal x whose reciprocal is normal
__device__ __forceinline__ double rcp64(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    r = fma(fma(-x, r, 1.0), r, r);
    return fma(fma(-x, r, 1.0), r, r);
}

// x / y from the reciprocal iy of y, to the last place (a remainder step):
// arguments of exponentials, whose rounding the exponential multiplies
__device__ __forceinline__ double div64(double x, double y, double iy)
{
    const double q = x * iy;
    return fma(fma(-q, y, x), iy, q);
}

// Linear short-characteristics weights over optical path d (sc_weights of the
// FP32 sweep, in FP64): e^{-d}, w_u, w_o and 1 - w_o, each without
// cancellation.  Below d = 1/2 from p = (d - 1 + e^{-d}) / d^2 = sum (-d)^n /
// (n+2)! (15 terms, truncation 6e-18) alone: w_o = d p, 1 - e^{-d} = d (1 -
// w_o); above, one exponential and one reciprocal.
__device__ __forceinline__ void sc64(double d, const double *__restrict__ tab, double &ex, double &wu, double &wo,
                                     double &omwo)
{
    if (d < 0.5) {
        double p = fma(d, 1.0 / 20922789888000.0, -1.0 / 1307674368000.0);
        p = fma(p, d, 1.0 / 87178291200.0);
        p = fma(p, d, -1.0 / 6227020800.0);
        p = fma(p, d, 1.0 / 479001600.0);
        p = fma(p, d, -1.0 / 39916800.0);
        p = fma(p, d, 1.0 / 3628800.0);
        p = fma(p, d, -1.0 / 362880.0);
        p = fma(p, d, 1.0 / 40320.0);
        p = fma(p, d, -1.0 / 5040.0);
        p = fma(p, d, 1.0 / 720.0);
        p = fma(p, d, -1.0 / 120.0);
        p = fma(p, d, 1.0 / 24.0);
        p = fma(p, d, -1.0 / 6.0);
        p = fma(p, d, 0.5);
        wo = d * p;
        omwo = 1.0 - wo;
        wu = d * (omwo - p);
        ex = fma(-d, omwo, 1.0);
    } else {
        ex = exp64(-d, tab);
        omwo = (1.0 - ex) * rcp64(d);
        wo = 1.0 - omwo;
        wu = omwo - ex;
    }
}

// H (and L where DISP) for a in [0, 0.05]
template <bool DISP>
__device__ __forceinline__ void voigt64(double a, double v, const double *__restrict__ tab, double &H, double &L)
{
    const double av = fabs(v);
    if (av < kV64Max) {
        const int j = (int)((float)av * (kV64N / (float)kV64Max));   // a neighbour's polynomial at its edge is as good
        const double *c = tab + min(j, kV64N - 1) * kV64Row;
        const double t = av - ((double)min(j, kV64N - 1) + 0.5) * (kV64Max / kV64N);
        double f = c[kV64Deg - 1], d = c[2 * kV64Deg - 1];
#pragma unroll
        for (int k = kV64Deg - 2; k >= 0; --k) {
            f = fma(f, t, c[k]);
            d = fma(d, t, c[kV64Deg + k]);
        }
        const double a2 = a * a, m2 = -2.0 * av;
        double D[10];
        D[0] = f;
        D[1] = d;
#pragma unroll
        for (int n = 1; n < 9; ++n) D[n + 1] = fma(m2, D[n], (-2.0 * n) * D[n - 1]);
        double o = fma(a2, D[9] * (1.0 / 362880), D[7] * (-1.0 / 5040));
        o = fma(o, a2, D[5] * (1.0 / 120));
        o = fma(o, a2, D[3] * (-1.0 / 6));
        o = fma(o, a2, D[1]);
        const double th2 = 4.0 * a2 * av * av;   // (2av)^2 <= 0.4 where e^{-v^2} counts
        // e^{a^2 - v^2}; a^2 <= 0.0025
        const double g = exp64(fma(a, a, -av * av), tab);
        double cs = fma(th2, 1.0 / 20922789888000.0, -1.0 / 87178291200.0);
        cs = fma(cs, th2, 1.0 / 479001600.0);
        cs = fma(cs, th2, -1.0 / 3628800.0);
        cs = fma(cs, th2, 1.0 / 40320.0);
        cs = fma(cs, th2, -1.0 / 720.0);
        cs = fma(cs, th2, 1.0 / 24.0);
        cs = fma(cs, th2, -0.5);
        cs = fma(cs, th2, 1.0);
        H = fma(g, cs, (-2.0 / 1.77245385090551602730 * a) * o);
        if (DISP) {
            double e = fma(a2, D[8] * (1.0 / 40320), D[6] * (-1.0 / 720));
            e = fma(e, a2, D[4] * (1.0 / 24));
            e = fma(e, a2, D[2] * -0.5);
            e = fma(e, a2, D[0]);
            double sn = fma(th2, -1.0 / 1307674368000.0, 1.0 / 6227020800.0);
            sn = fma(sn, th2, -1.0 / 39916800.0);
            sn = fma(sn, th2, 1.0 / 362880.0);
            sn = fma(sn, th2, -1.0 / 5040.0);
            sn = fma(sn, th2, 1.0 / 120.0);
            sn = fma(sn, th2, -1.0 / 6.0);
            sn = fma(sn, th2, 1.0);
            L = fma(2.0 / 1.77245385090551602730, e, -g * (2.0 * a * av) * sn);
            L = v < 0.0 ? -L : L;
        }
        return;
    }
    // w = (i / (sqrt(pi) z)) sum_k (2k-1)!! u^k, u = 1/(2z^2); the k-th term
    // over the first is below 1e-17 from k = K on
    // (e^{-v^2} < 2e-111 here)
    const int K = av < 24.0 ? 10 : (av < 60.0 ? 8 : 6);
    const double v2 = av * av, a2 = a * a;
    const double zr = 2.0 * (v2 - a2), zi = 4.0 * av * a;
    const double id = rcp64(fma(zr, zr, zi * zi));
    const double ur = zr * id, ui = -zi * id;
    const double *cf = tab + kT64Dfac;
    double sr = cf[K], si = 0.0;
    for (int k = K - 1; k >= 0; --k) {
        const double q = fma(sr, ur, fma(-si, ui, cf[k]));
        si = fma(sr, ui, si * ur);
        sr = q;
    }
    const double im = rcp64(1.77245385090551602730 * (v2 + a2));
    H = (sr * a - si * av) * im;
    if (DISP) L = (sr * av + si * a) * im;
    if (DISP) L = v < 0.0 ? -L : L;
}
#endif

}  // namespace rh
