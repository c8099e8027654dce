// Host tables of the pair kinematics, computed when a context is created (constants only: nothing here depends on a caller's
// data). Plain C++, no CUDA, so that a host program can check the entries. A(s) solves L(A) = coth A - 1/A = e^-s.
#pragma once

#include <cmath>
#include <cstddef>

namespace mcc {

// Table of the float pairs over x = ln s in [kN97X0, kN97X0 + kN97Nodes * kN97H].
constexpr int kN97Nodes = 512;
constexpr double kN97X0 = -6.907755278982137;  // ln 1e-3
constexpr double kN97X1 = 2.4849066497880004;  // ln 12
constexpr double kN97H = (kN97X1 - kN97X0) / kN97Nodes;

// Tables of the FP64 pairs (mcc_pair64.cuh).
constexpr int kF64N97 = 9 * 64;  // intervals of s: 64 per octave of [2^-5, 16); eight coefficients each of 1 / A(s), of
                                 // e^-2A (s < 2) or 1 - e^-2A, and of s A'(s) / A(s)
constexpr int kF64Turn = 256;    // (cos, sin) of multiples of 1/256 turn
constexpr int kF64Ln = 128;      // (r_i, -ln r_i)
constexpr size_t kF64TabDoubles = 24 * kF64N97 + 2 * kF64Turn + 2 * kF64Ln;

// L and dL/dA; below A = 3/2 from the power series of A coth A (radius pi), whose coefficients a_n follow from
// (A coth A) (sinh A / A) = cosh A.
template <class T>
void langevin(T A, T& L, T& dL)
{
    if (A >= T(1.5)) {
        const T sh = A < T(350) ? std::sinh(A) : T(1);
        L = 1 / std::tanh(A) - 1 / A;
        dL = 1 / (A * A) - (A < T(350) ? 1 / (sh * sh) : T(0));
        return;
    }
    constexpr int kTerms = 30;
    static const struct Series {
        T a[kTerms + 1];
        Series()
        {
            T fact[2 * kTerms + 2];
            fact[0] = 1;
            for (int n = 1; n < 2 * kTerms + 2; ++n) fact[n] = fact[n - 1] * n;
            for (int n = 0; n <= kTerms; ++n) {
                a[n] = 1 / fact[2 * n];
                for (int k = 0; k < n; ++k) a[n] -= a[k] / fact[2 * (n - k) + 1];
            }
        }
    } series;
    const T x2 = A * A;
    L = 0;
    dL = 0;
    for (int n = kTerms; n >= 1; --n) {
        L = L * x2 + series.a[n];
        dL = dL * x2 + (2 * n - 1) * series.a[n];
    }
    L *= A;
}

// One Newton step for A(s): on 1 - L(A) = 1 - e^-s for short lengths (1 - L = 1/A - 2/expm1(2A) keeps its relative
// precision), on L(A) = e^-s otherwise.
template <class T>
T n97_newton(T s, T A)
{
    T L, dL;
    langevin(A, L, dL);
    const T f = s < T(0.7) ? -std::expm1(-s) - (1 / A - 2 / std::expm1(2 * A)) : L - std::exp(-s);
    return A - f / dL;
}

// A(s): from the short-length series or the long-length inversion, Newton to double precision, then one step in the
// host's long double, so that the tables are correctly rounded up to an ulp.
inline long double n97_root(long double s)
{
    const double sd = (double)s, y = std::exp(-sd);
    double A = sd < 2.0 ? -1.0 / std::expm1(-sd) : 3.0 * y * (1.0 + 0.6 * y * y);
    for (int it = 0; it < 60; ++it) {
        double An = n97_newton(sd, A);
        if (!(An > 0.0)) An = 0.5 * A;
        if (An > 4.0 * A) An = 4.0 * A;
        const double d = std::fabs(An - A);
        A = An;
        if (d <= 1e-14 * A) break;
    }
    return n97_newton(s, (long double)A);
}

// Table of the float pairs: g = A s and h dg/dx (x = ln s) at the nodes.
inline void n97_table(float* g, float* dh)
{
    for (int k = 0; k <= kN97Nodes; ++k) {
        const double s = std::exp(kN97X0 + kN97H * k);
        const double A = (double)n97_root(s);
        double L, dL;
        langevin(A, L, dL);
        g[k] = (float)(A * s);  // d ln(A s)/dx = 1 - s e^-s / (A L'(A))
        dh[k] = (float)(A * s * kN97H * (1.0 - s * std::exp(-s) / (A * dL)));
    }
}

// cos of i / 256 turn, rounded once: the angle is brought to an eighth of a turn in whole numbers and its function taken in
// long double. (The cosine of a rounded double angle was off by up to 6e-16 and, next to a zero, by 77 units of the last
// place, which the pairs' azimuths and the normal deviates of TA77 inherited.)
inline double cos_turn(int i)
{
    const long double step = std::acos(-1.0L) / 128;
    i = (i % 256 + 256) % 256;
    if (i > 128) i = 256 - i;
    const bool neg = i > 64;
    if (neg) i = 128 - i;
    const double x = (double)(i <= 32 ? std::cos(i * step) : std::sin((64 - i) * step));
    return neg ? -x : x;
}

// Tables of mcc_pair64.cuh: Chebyshev interpolants of 1 / A(s), of e^-2A or 1 - e^-2A and of s A' / A as monomials in the
// interval's own variable t in [-1, 1], multiples of 1/256 turn, and the reciprocals and logarithms of mantissas in [0.6875, 1.375).
inline void f64_tables(double* out)
{
    constexpr int N = 8;
    using T = long double;
    T cosine[N][N], cheb[N][N];  // cosine[m][j] = T_m(node j); cheb[m]: monomial coefficients of T_m
    for (int m = 0; m < N; ++m) {
        for (int q = 0; q < N; ++q) cheb[m][q] = 0;
        if (m < 2) cheb[m][m] = 1;
        else
            for (int q = 0; q < N; ++q) cheb[m][q] = (q ? 2 * cheb[m - 1][q - 1] : T(0)) - cheb[m - 2][q];
        for (int j = 0; j < N; ++j) cosine[m][j] = std::cos(std::acos(T(-1)) * m * (2 * j + 1) / (2 * N));
    }
    for (int i = 0; i < kF64N97; ++i) {
        const T w = std::ldexp(T(1) / 64, i / 64 - 5);  // interval width
        const T a = std::ldexp(T(1), i / 64 - 5) + (i % 64) * w;
        T f[3][N];
        for (int j = 0; j < N; ++j) {
            const T s = a + w * (1 + cosine[1][j]) / 2, A = n97_root(s);
            f[0][j] = 1 / A;
            f[1][j] = i / 64 < 6 ? std::exp(-2 * A) : -std::expm1(-2 * A);  // s < 2; s >= 2
            T L, dL;
            langevin(A, L, dL);
            f[2][j] = -s * std::exp(-s) / (A * dL);  // s A' / A
        }
        for (int k = 0; k < 3; ++k) {
            T c[N] = {0, 0, 0, 0, 0, 0, 0, 0};
            for (int m = 0; m < N; ++m) {
                T b = 0;
                for (int j = 0; j < N; ++j) b += f[k][j] * cosine[m][j];
                b *= T(m ? 2 : 1) / N;
                for (int q = 0; q < N; ++q) c[q] += b * cheb[m][q];
            }
            for (int q = 0; q < N; ++q) out[N * (kF64N97 * k + i) + q] = (double)c[q];
        }
    }
    double* turn = out + 3 * N * kF64N97;
    for (int i = 0; i < kF64Turn; ++i) {
        turn[2 * i] = cos_turn(i);
        turn[2 * i + 1] = cos_turn(i - kF64Turn / 4);
    }
    double* ln = turn + 2 * kF64Turn;
    for (int i = 0; i < kF64Ln; ++i) {  // mantissas below 1 come in steps of 1/256, above in steps of 1/128
        const double m = i < 80 ? 0.6875 + (i + 0.5) / 256.0 : 1.0 + (i - 80 + 0.5) / 128.0;
        const double r = i == 79 || i == 80 ? 1.0 : (double)(float)(1.0 / m);
        ln[2 * i] = r;
        ln[2 * i + 1] = r == 1.0 ? 0.0 : (double)-std::log((T)r);
    }
}

}  // namespace mcc
