// FP64 kinematics of one scattering pair: the N97 / TA77 angle, the azimuth and the rotation, shared by the one-CTA step
// kernel and the adjoint.
//
// The FP64 pipe bounds both (GB300 issues FP64 at 1/64 of the float rate; it was 81% busy while an SM worked), and most
// of its instructions were the pair's: two Newton steps on the N97 root (expm1, sinh, three divisions each), expm1,
// log1p, log, exp, sincospi and eight divisions, about 600 FP64 instructions per pair. Here the functions whose
// arguments are known in form are table lookups with a short series, each within about an ulp:
//   1 / A(s)    piecewise degree-7 polynomials in s (64 per octave of [2^-5, 16)); below, the series of 1 - e^-s, which
//               equals 1 / A there to 1e-27; above, the inversion of L(A) = A/3 - A^3/45
//   e^-2A       the same intervals: e^-2A below s = 2, 1 - e^-2A above (the smaller one, or nearly). Its polynomials lose
//               relative precision towards s = 2^-5, where e^-2A is below 1e-16 of what it is added to
//   ln u        u = 2^k m, ln m = -ln r_i + ln(m r_i) with tabulated r_i ~ 1/m (Tang, "Table-driven implementation of
//               the logarithm function in IEEE floating-point arithmetic", 1990); mantissas in [0.6875, 1.375), 128
//               intervals and r_i = 1 next to 1 are the arrangement of the public log of Arm's Optimized Routines (the
//               reciprocals, the logarithms and the Taylor terms are computed here);
//               one logarithm per pair: of whichever of 1 - cos and 1 + cos is smaller, the other being 2 minus it
//   azimuth     2 pi (k + 1/2) 2^-23 = nearest 1/256 turn, tabulated, + a remainder below pi/256 (addition theorem)
// uniforms are assembled from their bits instead of converted, and comparisons are made on the bits (an FP64 comparison
// takes the FP64 pipe too). Roots and quotients taken through reciprocals get one correction from their exactly formed residual, so
// a pair's velocity change is as close to extended precision as the same formulas in plain double (rms 1.5e-16 of itself for N97,
// 1.9e-16 for TA77; uncorrected 1.9e-16 and 2.2e-16). About 130 instructions per pair. FP64 step of 4096
// three-species cells (2.1e6 particles) 6.11 -> 2.13 ms, relativistic beam of 2048 cells 6.45 -> 2.01 ms (2.06 and 1.93 without
// the corrections); error against 64-bit results 1.3e-16 of the velocities.
#pragma once

#include "mcc_kernels.h"

namespace mcc {

// Uniform on (0, 1): ((r >> 9) + 1/2) 2^-23.
__device__ __forceinline__ double u23_bits(uint32_t r)
{
    return __hiloint2double((int)(0x3FF00000u | (r >> 12)), (int)(((r << 20) & 0xE0000000u) | 0x10000000u)) - 1.0;
}

// cos and sin of 2 pi ((r >> 9) + 1/2) 2^-23: the nearest 1/256 turn plus the remainder. The zeros of both are table entries,
// so a result next to a zero keeps its relative precision (TA77 multiplies it by the root of a large s).
__device__ __forceinline__ void turn64(const F64Tab& T, uint32_t r, double& cs, double& sn)
{
    const uint32_t up = (r >> 23) & 1u;  // past the middle of the 1/256 turn: the next entry is nearer
    const double2 a = __ldg(T.turn + (((r >> 24) + up) & 255u));  // cos, sin
    const double m = __hiloint2double((int)(0x3FF00010u | ((r >> 4) & 0xFFFE0u)), 0);  // 1 + position within it
    const double d = (m - (up ? 2.0 : 1.0)) * 0.02454369260617025968;                   // 2 pi / 256
    const double d2 = d * d;
    const double sd = d * fma(d2, fma(d2, fma(d2, -1.0 / 5040.0, 1.0 / 120.0), -1.0 / 6.0), 1.0);
    const double cm = d2 * fma(d2, fma(d2, -1.0 / 720.0, 1.0 / 24.0), -0.5);
    cs = a.x + fma(a.x, cm, -a.y * sd);
    sn = a.y + fma(a.y, cm, a.x * sd);
}

// ln(u + c) for a positive normal u and a c below its rounding (to first order).
__device__ __forceinline__ double ln64(const F64Tab& T, double u, double c)
{
    const int hi = __double2hiint(u);
    const int ix = hi - 0x3FE60000;  // mantissas are taken in [0.6875, 1.375)
    const int k = ix >> 20;
    const double2 t = __ldg(T.ln + ((ix >> 13) & 127));  // r_i, -ln r_i
    const double m = __hiloint2double(hi - (k << 20), __double2loint(u));
    const double f = fma(m, t.x, -1.0);  // |f| < 0.008; r_i = 1 in the two intervals next to 1
    double p = fma(f, -1.0 / 8.0, 1.0 / 7.0);
    p = fma(f, p, -1.0 / 6.0);
    p = fma(f, p, 1.0 / 5.0);
    p = fma(f, p, -1.0 / 4.0);
    p = fma(f, p, 1.0 / 3.0);
    p = fma(f, p, -0.5);
    // c / u with 2^-k r_i for 1 / u
    const double ru = __hiloint2double(__double2hiint(t.x) - (k << 20), __double2loint(t.x));
    const double l = fma(f * f, p, fma(c, ru, f));
    // k converted exactly by an addition
    const double kd = __hiloint2double(0x43300000, (int)(0x80000000u ^ (uint32_t)k)) - 4503601774854144.0;
    return fma(kd, 0.69314718055994530942, t.y + l);
}

// Polynomial of one interval of s in [2^-5, 16): coefficients at tab[4 k ..] for interval k.
__device__ __forceinline__ double n97_poly(const double2* tab, double s)
{
    const int hi = __double2hiint(s);
    const double2* c = tab + 4 * ((hi >> 14) - (0x3FA00000 >> 14));
    const double m = __hiloint2double(0x3FF00000 | (hi & 0x3FFF), __double2loint(s));
    const double t = fma(m, 128.0, -129.0);  // [-1, 1) over the interval
    const double2 c0 = __ldg(c), c1 = __ldg(c + 1), c2 = __ldg(c + 2), c3 = __ldg(c + 3);
    double p = fma(t, c3.y, c3.x);
    p = fma(t, p, c2.y);
    p = fma(t, p, c2.x);
    p = fma(t, p, c1.y);
    p = fma(t, p, c1.x);
    p = fma(t, p, c0.y);
    return fma(t, p, c0.x);
}

// 1 / A(s) of the N97 angle, s > 0, and with EF e^-2A and 1 - e^-2A (A > 31 below s = 2^-5: e^-2A < 1e-27 counts as 0).
template <bool EF>
__device__ __forceinline__ double n97_rA(const F64Tab& T, double s, double& E, double& F)
{
    const int hi = __double2hiint(s);
    if (hi < 0x3FA00000) {  // s < 2^-5
        if (EF) {
            E = 0.0;
            F = 1.0;
        }
        double p = fma(s, -1.0 / 40320.0, 1.0 / 5040.0);
        p = fma(s, p, -1.0 / 720.0);
        p = fma(s, p, 1.0 / 120.0);
        p = fma(s, p, -1.0 / 24.0);
        p = fma(s, p, 1.0 / 6.0);
        p = fma(s, p, -0.5);
        return fma(s * s, p, s);
    }
    if (hi >= 0x40300000) {  // s >= 16: A < 4e-7
        const double y = exp(-s);
        const double A = 3.0 * y * fma(0.6 * y, y, 1.0);
        if (EF) {
            const double t = A + A;
            F = t * fma(t, fma(t, 1.0 / 6.0, -0.5), 1.0);
            E = 1.0 - F;
        }
        return 1.0 / A;
    }
    if (EF) {
        const double h = n97_poly(T.n97 + 4 * kF64N97, s);
        const double r = 1.0 - h;
        E = hi < 0x40000000 ? h : r;
        F = hi < 0x40000000 ? r : h;
    }
    return n97_poly(T.n97, s);
}

// A(s) for sample_angle: 0 where 1 - e^-s rounds to 1 or s is not a number (isotropic), infinite for s <= 0 (no scattering).
__device__ __forceinline__ double n97_A(double s, const F64Tab& T)
{
    double E, F;
    if (!(s <= 36.7)) return 0.0;
    return s > 0.0 ? 1.0 / n97_rA<false>(T, s, E, F) : CUDART_INF;
}

// x >= the value whose high word is lo, from the high word of x; false for NaN.
__device__ __forceinline__ bool from64(int hi, int lo) { return (uint32_t)(hi - lo) <= (uint32_t)(0x7FF00000 - lo); }

// s A'(s) / A(s), the logarithmic derivative of the N97 root, s > 0.
__device__ __forceinline__ double n97_W(const F64Tab& T, double s)
{
    const int hi = __double2hiint(s);
    if (hi < 0x3FA00000) {  // -s / (e^s - 1)
        const double s2 = s * s;
        return fma(s2, fma(s2, fma(s2, -1.0 / 30240.0, 1.0 / 720.0), -1.0 / 12.0), fma(0.5, s, -1.0));
    }
    if (hi >= 0x40300000) {  // A = 3 y (1 + 3 y^2 / 5), y = e^-s
        const double y = exp(-s);
        return -s * fma(1.2 * y, y, 1.0);
    }
    return n97_poly(T.n97 + 8 * kF64N97, s);
}

// Polar angle of a pair, sin(Theta) and 1 - cos(Theta), from the scattering length s and the draws (r.x, r.w).
// DERIV and want: also s times their derivatives in s.
//  TA77: tan(Theta/2) = d = sqrt(s/2) g, g normal by Box-Muller; sin = 2 d / (1 + d^2), 1 - cos = 2 d^2 / (1 + d^2).
//  N97:  1 - cos = -ln((1 - U) + U e^-2A) / A, 1 + cos = ln1p((1 - U) expm1(2A)) / A; s above 36.7 is isotropic. What 1 - e^-s
//        says beyond (as on the mixed path): no scattering for a negative s, isotropic if s is not a number.
// The products whose rounding the two callers have to share are kept from being contracted.
template <bool DERIV>
__device__ __forceinline__ void angle64(const F64Tab& T, int method, double s, const uint4& r, double& st, double& omc,
                                        bool want, double& sdst, double& sdomc)
{
    const double U = u23_bits(r.x);
    if (DERIV) sdst = sdomc = 0.0;
    if (method == 0) {
        double cs, sn;
        turn64(T, r.w, cs, sn);
        const double t = -s * ln64(T, U, 0.0);  // bounded so that d^2 is finite
        const double d = sqrt(from64(__double2hiint(t), 0x6974E718) ? 1e200 : t) * cs;
        const double d2 = __dmul_rn(d, d), q = 1.0 / (1.0 + d2);
        st = 2.0 * d * q;
        omc = 2.0 * d2 * q;
        if (DERIV && want) {  // s d' = d / 2
            const double x = q * q;
            sdst = d * (1.0 - d2) * x;
            sdomc = 2.0 * d2 * x;
        }
        return;
    }
    const double V = 1.0 - U;  // exact
    double o, q;
    const int hs = __double2hiint(s);
    const uint32_t as = (uint32_t)hs & 0x7FFFFFFFu;
    if (as >= 0x40425800u && (hs >= 0 || as > 0x7FF00000u)) {  // s >= 36.69 or not a number: isotropic
        o = 2.0 * U;
        q = 2.0 * V;
    } else if (hs < 0) {  // s < 0, from a negative Coulomb logarithm: no scattering
        o = 0.0;
        q = 2.0;
    } else {
        double E, F;  // e^-2A, 1 - e^-2A
        const double rA = n97_rA<true>(T, s, E, F);
        // 1 - cos = -ln(1 + x) / A, x = -U F: 1 + x itself while |x| is below 1/2, the two positive terms (1 - U) + U E
        // beyond. Where that exceeds 1, 1 + cos = ln(1 + y) / A, y = (1 - U) (e^2A - 1), takes its place.
        const double x = __dmul_rn(-U, F);
        const bool near1 = (__double2hiint(x) & 0x7FFFFFFF) < 0x3FE00000;
        const double u = near1 ? 1.0 + x : fma(U, E, V);
        const bool far = __double_as_longlong(u * u) < __double_as_longlong(E);  // 1 + x < e^-A
        double z = x, a = u;
        if (far) {
            // s < 1/8 gets here with probability below e^-8: e^-2A from the exponential, in full relative precision
            if (hs < 0x3FC00000) E = exp(-2.0 / rA);
            z = __dmul_rn(V, F / E);
            a = 1.0 + z;
        }
        const double l = __dmul_rn(ln64(T, a, near1 || far ? z - (a - 1.0) : 0.0), rA);
        o = far ? 2.0 - l : -l;
        q = far ? l : 2.0 + l;
        if (DERIV && want) {
            // d(1 - cos)/dA = (-(1 - cos) + 2 U E / (1 + x)) / A
            sdomc = (2.0 * U * E / u - o) * n97_W(T, s);
            const double p = o * q;
            sdst = p > 0.0 ? (q - o) * sdomc * (0.5 * rsqrt(p)) : 0.0;
            if (from64(__double2hiint(o), 0x40000000)) sdomc = sdst = 0.0;
        }
    }
    o = from64(__double2hiint(o), 0x40000000) ? 2.0 : o;
    q = from64(__double2hiint(q), 0x40000000) ? 2.0 : q;
    omc = o;
    st = sqrt(o * q);
}

// sqrt(x) from r = rsqrt(x), with one correction from the exactly formed residual x - y^2: half a unit of the last place, where
// x r alone is off by up to one and a half. Two instructions instead of the dozen of a square root.
__device__ __forceinline__ double root64(double x, double r)
{
    const double y = x * r;
    return fma(fma(-y, y, x), 0.5 * r, y);
}

// Rotation of u (magnitude um) through (Theta, phi) about its own direction; returns du = u' - u.
__device__ __forceinline__ void rotate64(double ux, double uy, double uz, double um, double st, double omc, double cp,
                                         double sp, double& dx, double& dy, double& dz)
{
    const double p2 = fma(ux, ux, uy * uy);
    const double sc = st * cp, ss = st * sp;
    if (p2 > 0.0) {
        const double rp = rsqrt(p2);
        const double ax = ux * rp, ay = uy * rp;
        const double zc = uz * sc, us = um * ss;
        dx = ax * zc - ay * us - ux * omc;
        dy = ay * zc + ax * us - uy * omc;
        dz = -root64(p2, rp) * sc - uz * omc;
    } else {
        dx = um * sc;
        dy = um * ss;
        dz = -uz * omc;
    }
}

// Change of the relative velocity u = v_i - v_j of a non-relativistic pair, s = cw / |u|^3; false if u vanishes. cw = kappa
// / mu^2 w_max N_min, halved for a triplet. The step kernel and the adjoint's forward both run this and then fma(mu / m, du,
// v), so that a replayed interaction repeats the step's velocities bit for bit.
// TAPE and pt: what the reverse of the pair reads goes to pt, one value every n: u = v_i - v_j (3), 1 / |u|, sin(Theta),
// 1 - cos(Theta), s times their derivatives in s, cos(phi), sin(phi).
constexpr int kPairTape = 10;
template <bool TAPE>
__device__ __forceinline__ bool pair64(const F64Tab& T, int method, double cw, const double vi[3], const double vj[3],
                                       const uint4& r, double du[3], double* pt = nullptr, size_t n = 0)
{
    const double ux = vi[0] - vj[0], uy = vi[1] - vj[1], uz = vi[2] - vj[2];
    const double u2 = fma(uz, uz, fma(uy, uy, ux * ux));
    if (__double_as_longlong(u2) == 0) return false;
    const double ru = rsqrt(u2), um = root64(u2, ru);
    // 1 / |u|^3: ru^3 (three roundings over three times that of ru), corrected once
    const double u3 = u2 * um, r3 = ru * ru * ru;
    double st, omc, sp, cp, d0, d1;
    angle64<TAPE>(T, method, cw * fma(fma(-u3, r3, 1.0), r3, r3), r, st, omc, pt != nullptr, d0, d1);
    turn64(T, r.y, cp, sp);
    if (TAPE && pt) {
        const double x[kPairTape] = {ux, uy, uz, ru, st, omc, d0, d1, cp, sp};
#pragma unroll
        for (int k = 0; k < kPairTape; ++k) pt[k * n] = x[k];
    }
    rotate64(ux, uy, uz, um, st, omc, cp, sp, du[0], du[1], du[2]);
    return true;
}

// The coefficients of a correction in double, shared by the step kernel and the adjoint's forward. Every product and sum is rounded
// as written (the compiler contracts a product into a sum differently in the two kernels, and the crossing pairs' last bits
// then differ).
// m_a x_a + m_b x_b (the first alone for one species).
__device__ __forceinline__ double mass_sum(double ma, double xa, double mb, double xb, bool intra)
{
    return fma(ma, xa, intra ? 0.0 : __dmul_rn(mb, xb));
}
// A species' weight in the split of Delta E (Eq. DeltaEs): mean weight times post-shift energy.
__device__ __forceinline__ double split_weight64(double W1, int n, double E) { return __dmul_rn(W1 / (double)n, E); }
// Delta E split between species a and b of weights wa and wb: a species with fewer than two particles takes no share. Returns 1 if
// no species can take it.
__device__ __forceinline__ int split64(bool intra, int na, int nb, double wa, double wb, double dE, double& D0, double& D1)
{
    D0 = dE;
    D1 = 0.0;
    if (intra) return 0;
    const bool can0 = na >= 2, can1 = nb >= 2;
    if (can0 && can1) {
        const double den = __dadd_rn(wa, wb);
        if (!(den > 0.0)) return dE != 0.0;
        D0 = __dmul_rn(wa / den, dE);
        D1 = __dsub_rn(dE, D0);
    } else if (can1) {
        D0 = 0.0;
        D1 = dE;
    } else if (!can0) {
        return dE != 0.0;
    }
    return 0;
}

// Momentum change of particle i of a relativistic pair in the lab frame (proper velocities vi, vj, masses ma, mb): the
// pair's centre-of-momentum frame (see rel_cm), s with |p*|^2 v_rel* in place of mu^2 u^3, the rotation of p* and the
// boost of its change back. kw = kappa w_max N_min (halved for a triplet). False if p* vanishes.
__device__ __forceinline__ bool rel_pair64(const F64Tab& T, int method, double c2, double ma, double mb, double kw,
                                           const double vi[3], const double vj[3], const uint4& r, double dp[3])
{
    const double ic2 = 1.0 / c2;
    const double gi = sqrt(fma(vi[0] * vi[0] + vi[1] * vi[1] + vi[2] * vi[2], ic2, 1.0));
    const double gj = sqrt(fma(vj[0] * vj[0] + vj[1] * vj[1] + vj[2] * vj[2], ic2, 1.0));
    const double M = ma * gi + mb * gj, rM = 1.0 / M;
    double du[3], V[3], du2 = 0.0, ss = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        du[d] = vi[d] - vj[d];
        V[d] = (ma * vi[d] + mb * vj[d]) * rM;
        du2 += du[d] * du[d];
        ss += du[d] * (vi[d] + vj[d]);
    }
    const double dg = ss * ic2 / (gi + gj);
    const double grm1 = fmax(0.5 * (du2 * ic2 - dg * dg), 0.0);
    const double sm = ma + mb;
    const double gC = M * rsqrt(fma(sm, sm, 2.0 * ma * mb * grm1));
    const double cb = gC * gC * ic2 / (gC + 1.0);
    const double k = ma * mb * rM;
    double p[3], Vq = 0.0, p2 = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        p[d] = k * (gj * du[d] - dg * vj[d]);
        Vq += V[d] * p[d];
    }
    Vq *= cb;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        p[d] = fma(Vq, V[d], p[d]);
        p2 += p[d] * p[d];
    }
    if (!(p2 > 0.0)) return false;
    const double pm = root64(p2, rsqrt(p2));
    // v_rel* = |p*| (1 / (m_a gamma_a*) + 1 / (m_b gamma_b*)), m gamma* = sqrt(m^2 + |p*|^2 / c^2)
    const double pc = p2 * ic2;
    const double iv = rsqrt(fma(ma, ma, pc)) + rsqrt(fma(mb, mb, pc));
    const double s = kw / (p2 * pm * iv);
    double st, omc, cp, sp, x0, x1, d[3];
    angle64<false>(T, method, s, r, st, omc, false, x0, x1);
    turn64(T, r.y, cp, sp);
    rotate64(p[0], p[1], p[2], pm, st, omc, cp, sp, d[0], d[1], d[2]);
    const double Vd = cb * (V[0] * d[0] + V[1] * d[1] + V[2] * d[2]);
#pragma unroll
    for (int q = 0; q < 3; ++q) dp[q] = fma(Vd, V[q], d[q]);
    return true;
}

}  // namespace mcc
