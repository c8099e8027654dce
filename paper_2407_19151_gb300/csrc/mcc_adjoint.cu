// Pathwise adjoint of one interaction of the collision step (FP64, non-relativistic), for gradients of a loss of the
// final velocities with respect to the initial velocities, the weights and the Coulomb logarithm.
//
// Every random draw and every discrete decision of the step is held fixed: the Philox draws, the permutations and
// TA77 pairs, the accept test of the heavier particle (Sec. 3.2), the weight order, the energy-correction pass
// structure and the crossing pair (the one that absorbs the remainder of Delta E_s). Between those decisions the
// interaction is a smooth map  v_before -> v_after  with parameters w and lnL:
//   scatter  (Sec. 3.2, Eq. sab_TA77): s = kappa lnL w_max N_min / (mu^2 u^3), N97 A(s) from coth A - 1/A = e^-s or
//            TA77 delta = sqrt(s/2) g, the polar angle, the rotation of u, the lighter/heavier updates;
//   shift    (Eq. vp_pm): v_pm = v_ps - B w, B = sum m w (v_ps - v_bs) / sum m w^2;
//   Delta E  (Eq. Econs, Eq. DeltaEs): per-particle energy differences, split by mean weight x post-shift energy;
//   energy pairs (Eqs. vp1/vp2/vrel_inelastic, U_inelastic): capped pairs U = sign(D) fE K, the crossing pair
//            U = D - (sum of the earlier pairs' U); v1' = v1 + m2/M (g - 1) v_R, v2' = v2 - m1/M (g - 1) v_R,
//            g = sqrt(1 - U/K);
//   rollback (Sec. 5.2) when the correction fails: v_after = v_before.
// A Delta E_s that vanishes (equal weights, or below the rounding-noise threshold) is differentiated as its limit:
// the first pair of the order as the crossing pair with U = Delta E_s = 0.
// The kernel recomputes the interaction from the stored pre-interaction state, keeping a tape of every pair's angles,
// then runs the chain rule backwards through the tape (one CTA per cell; the tape in a per-CTA slab of the workspace).
// With a recorded tape the slabs are per cell and outlive the call: a recording call runs the forward and keeps each
// cell's slab (the tape and the per-cell scalars of the correction); a later replaying call on the same interaction
// runs only the reverse sweep from it.
//
// What bounds it: the FP64 pipe for the pairs (mcc_pair64.cuh), once the serial parts are out of the way. The working
// arrays that are read in random order (state or gradient, weights, sort keys, permutation, weight order: 64 B per
// particle) live in shared memory, the permutations are counting sorts there, and both directions of the energy pairs
// run 32 at a time (a pass's pairs are disjoint; the forward needs a prefix sum over their caps, the reverse only the
// crossing pair's dL/dU, which comes first). Two recorded steps of 1024 cells x 512 with their reverse: 5.9 -> 2.3 ms
// (3.8 with the pair functions alone, 2.6 before the pairs' angles were taped with their derivatives). The forward sums
// what the step kernel sums in its order, so a replay from a checkpoint repeats the step's trajectory bit for bit (the
// closed-form gradients over 50 steps from checkpoints then hold as closely as from tapes, 1e-11 where they held 3e-10).
#include "mcc_pair64.cuh"
#include "mcc_perm.cuh"

namespace mcc {
namespace {

constexpr int kAdjCtasPerSm = 4;  // resident CTAs the kernel's registers are bounded for

constexpr int kFlagUpdI = 1 << 28, kFlagUpdJ = 1 << 29, kFlagActive = 1 << 30, kPairIndex = kFlagUpdI - 1;

struct AdjArgs {
    StepArgs a;                // state before the interaction (vx, vy, vz: double), w, constants of ic[0]
    double lnL;                // Coulomb logarithm of the interaction
    double* ox;                // state after the interaction (null: not written)
    double* oy;
    double* oz;
    double* gx;                // in: dL/dv after; out: dL/dv before (null: forward only)
    double* gy;
    double* gz;
    double* gw;                // += dL/dw
    double* glnL;              // += dL/dlnL (one value)
    char* slab;
    int64_t slab_stride;
    int32_t max_cell;
    int32_t max_epairs;
    int32_t tape;              // 0: per-CTA slabs, recompute; 1: per-cell slabs, record; 2: per-cell slabs, replay
    int32_t on_chip;           // working arrays in shared memory (else in the slab)
};

// Per-cell scalars of the forward that the reverse sweep reads (kept at the end of a recorded slab).
struct TapeHead {
    int fail, ne[2], e0[2], zeroed[2];
    double B[3], Sw, S[3], dE, Es[2], W1[2], D[2];
};

// The tape of one cell (n = max_cell, E = max_epairs).
struct Slab {
    double* vb;     // [3][n] before the interaction
    double* vm;     // [3][n] after the momentum shift
    double* pv;     // [kPairTape][n] per scatter pair, see pair64
    double* ev;     // [6][E] per energy pair: v_1, v_2 at the pair's turn
    double* eU;     // [E]
    double* eK;     // [E]
    int32_t* pi;    // [n] scatter pair particles; the flags in the top bits of the first
    int32_t* pj;
    int32_t* ei;    // [E] energy pair particles; 2 pass + (1 if the pair took its cap)
    int32_t* ej;
    int32_t* ecap;
    TapeHead* head;
    char* work;     // working arrays of cells too large for shared memory
    int n, E;
};

// Working arrays of the cell in progress: the forward's and, over the same bytes, the reverse sweep's.
struct Work {
    double* v;       // [3][n] forward: the state; reverse: gradient of the current stage
    uint64_t* keys;  // [n] forward: sort keys
    double* gwl;     // [n] reverse: dL/dw of this interaction (over keys)
    uint32_t* cnt;   // [2 n] forward: bucket counters
    int32_t* perm;   // [n] forward: random permutation (cell-local indices, segment start included)
    int32_t* rho;    // [n] forward: energy-pair order
    double* gb;      // [3][n] reverse: gradient reaching v_before directly through the correction (over cnt ..)
    double* w;       // [n] weights
};
constexpr size_t kWorkBytesPerParticle = 24 + 8 + 24 + 8;

__device__ __forceinline__ Work make_work(char* base, int n)
{
    Work k;
    k.v = reinterpret_cast<double*>(base);
    k.gwl = k.v + 3 * (size_t)n;
    k.keys = reinterpret_cast<uint64_t*>(k.gwl);
    k.gb = k.gwl + n;
    k.cnt = reinterpret_cast<uint32_t*>(k.gb);
    k.perm = reinterpret_cast<int32_t*>(k.gb + n);
    k.rho = k.perm + n;
    k.w = k.gb + 3 * (size_t)n;
    return k;
}

__host__ __device__ inline size_t al8(size_t x) { return (x + 7) & ~(size_t)7; }

__host__ __device__ inline size_t slab_bytes(int n, int E, bool on_chip)
{
    const size_t dn = (size_t)n, de = (size_t)E;
    return 2 * al8(24 * dn) + al8(8 * kPairTape * dn) + al8(48 * de) + 2 * al8(8 * de) + 2 * al8(4 * dn) + 3 * al8(4 * de) +
           al8(sizeof(TapeHead)) + (on_chip ? 0 : kWorkBytesPerParticle * dn) + 256;
}

__device__ Slab make_slab(char* base, int n, int E)
{
    Slab s;
    s.n = n;
    s.E = E;
    size_t o = 0;
    auto take = [&](size_t b) {
        char* p = base + o;
        o += al8(b);
        return p;
    };
    s.vb = reinterpret_cast<double*>(take(24 * (size_t)n));
    s.vm = reinterpret_cast<double*>(take(24 * (size_t)n));
    s.pv = reinterpret_cast<double*>(take(8 * kPairTape * (size_t)n));
    s.ev = reinterpret_cast<double*>(take(48 * (size_t)E));
    s.eU = reinterpret_cast<double*>(take(8 * (size_t)E));
    s.eK = reinterpret_cast<double*>(take(8 * (size_t)E));
    s.pi = reinterpret_cast<int32_t*>(take(4 * (size_t)n));
    s.pj = reinterpret_cast<int32_t*>(take(4 * (size_t)n));
    s.ei = reinterpret_cast<int32_t*>(take(4 * (size_t)E));
    s.ej = reinterpret_cast<int32_t*>(take(4 * (size_t)E));
    s.ecap = reinterpret_cast<int32_t*>(take(4 * (size_t)E));
    s.head = reinterpret_cast<TapeHead*>(take(sizeof(TapeHead)));
    s.work = base + o;
    return s;
}

struct AdjShared {
    int off[kMaxSpecies + 1];
    int fail, fail0;  // the correction failed; no species could take a share
    int ne[2];        // energy pairs taped per side
    int e0[2];        // first tape entry of each side
    int zeroed[2];    // Delta E_s set to zero as rounding noise
    double B[3], Sw, S[3];
    double dE, Es[2], W1[2], D[2], gD[2], gB[3];
    double gS[3], gSw, gdE, gEs[2], gW1[2];
    int iscan[kWarps + 1];
    alignas(16) unsigned char red_raw[8 * kThreads * 8];
    alignas(8) unsigned char red[8 * 8];
};

__device__ __forceinline__ Acc<double>* accp(unsigned char* p) { return reinterpret_cast<Acc<double>*>(p); }

// Forward of one scatter pair (the FP64 pair loop of the step kernel); returns the flags. pt: its tape (null: none).
__device__ int pair_forward(const StepArgs& A, const InterConst& ic, double vi[3], double vj[3], double wi, double wj,
                            int nmin, bool trip, uint4 r, double* pt, size_t n)
{
    int flags = 0;
    bool upd_i = true, upd_j = true;
    if (wi != wj) {
        const bool moves = u23_bits(r.z) * fmax(wi, wj) < fmin(wi, wj);
        if (wi > wj) upd_i = moves;
        else upd_j = moves;
    }
    if (upd_i) flags |= kFlagUpdI;
    if (upd_j) flags |= kFlagUpdJ;
    const double wf = (wi > wj ? wi : wj) * (double)nmin;
    double du[3];
    if (!pair64<true>(A.t64, A.method, (trip ? 0.5 : 1.0) * ic.kappa_mu2 * wf, vi, vj, r, du, pt, n)) return flags;
    flags |= kFlagActive;
    for (int k = 0; k < 3; ++k) {
        if (upd_i) vi[k] = fma(ic.mu_ma, du[k], vi[k]);
        if (upd_j) vj[k] = fma(-ic.mu_mb, du[k], vj[k]);
    }
    return flags;
}

// Reverse of one scatter pair from its tape (at pv, one value every N): g1, g2 (dL/d outputs) -> dL/d inputs in place;
// dL/dw of the heavier particle accumulated; returns s dL/ds (not a number for lnL = 0: s carries no derivative in it
// then). The angles are taped with their derivatives: taking them again cost more than half of the sweep's FP64
// instructions (two recorded steps of 1024 cells x 512 with their reverse: 2.62 -> 2.30 ms).
__device__ double pair_reverse(const InterConst& ic, double lnL, const double* pv, int N, double wi, double wj,
                               int flags, double g1[3], double g2[3], double& gwi, double& gwj)
{
    if (!(flags & kFlagActive)) return 0.0;
    const double fa = (flags & kFlagUpdI) ? ic.mu_ma : 0.0, fb = (flags & kFlagUpdJ) ? ic.mu_mb : 0.0;
    const double gd[3] = {fa * g1[0] - fb * g2[0], fa * g1[1] - fb * g2[1], fa * g1[2] - fb * g2[2]};
    if (gd[0] == 0.0 && gd[1] == 0.0 && gd[2] == 0.0) return 0.0;
    const double u[3] = {pv[0], pv[N], pv[2 * (size_t)N]};
    const double ru = pv[3 * (size_t)N], st = pv[4 * (size_t)N], omc = pv[5 * (size_t)N];
    const double cp = pv[8 * (size_t)N], sp = pv[9 * (size_t)N];
    const double um = (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]) * ru;
    // rotation du(u, st, omc) backwards
    double gst, gu[3], gum;
    const double gomc = -(gd[0] * u[0] + gd[1] * u[1] + gd[2] * u[2]);
    const double up2 = u[0] * u[0] + u[1] * u[1];
    const double uc = u[2] * cp, us = um * sp, tc = st * cp, ts = st * sp;
    if (up2 > 0.0) {
        const double rp = rsqrt(up2);
        const double a = u[0] * rp, b = u[1] * rp;
        const double g01 = gd[0] * a + gd[1] * b, g10 = gd[1] * a - gd[0] * b;
        gst = g01 * uc + g10 * us - gd[2] * (up2 * rp) * cp;
        gum = g10 * ts;
        const double x = u[2] * tc, y = um * ts;
        const double ga = gd[0] * x + gd[1] * y, gb = gd[1] * x - gd[0] * y;
        const double gup = -gd[2] * tc - (ga * a + gb * b) * rp;
        gu[0] = ga * rp + gup * a - gd[0] * omc;
        gu[1] = gb * rp + gup * b - gd[1] * omc;
        gu[2] = g01 * tc - gd[2] * omc;
    } else {
        gst = (gd[0] * cp + gd[1] * sp) * um;
        gum = gd[0] * tc + gd[1] * ts;
        gu[0] = 0.0;
        gu[1] = 0.0;
        gu[2] = -gd[2] * omc;
    }
    // angle, then s = C w_max / um^3
    const double gss = gst * pv[6 * (size_t)N] + gomc * pv[7 * (size_t)N];
    gum = (gum - 3.0 * gss * ru) * ru;
    for (int k = 0; k < 3; ++k) {
        const double x = fma(gum, u[k], gu[k]);
        g1[k] += x;
        g2[k] -= x;
    }
    if (wi > wj) gwi += gss / wi;
    else gwj += gss / wj;
    return lnL == 0.0 ? CUDART_NAN : gss;
}

__device__ __forceinline__ void ld3(const double* p, int n, int i, double x[3])
{
    x[0] = p[i];
    x[1] = p[n + i];
    x[2] = p[2 * n + i];
}
__device__ __forceinline__ void st3(double* p, int n, int i, const double x[3])
{
    p[i] = x[0];
    p[n + i] = x[1];
    p[2 * n + i] = x[2];
}

// k-th TA77 pair (cell-local indices) with p mod N_min supplied (inter).
__device__ __forceinline__ void pair_of(const int32_t* perm, bool intra, int na, int nb, int a0, int b0, int p, int pm,
                                        int& i, int& j, bool& trip)
{
    trip = false;
    if (intra) {
        if (na & 1) {
            if (p < 3) {
                i = perm[a0 + p];
                j = perm[a0 + (p + 1) % 3];
                trip = true;
                return;
            }
            i = perm[a0 + 2 * p - 3];
            j = perm[a0 + 2 * p - 2];
            return;
        }
        i = perm[a0 + 2 * p];
        j = perm[a0 + 2 * p + 1];
        return;
    }
    if (na >= nb) {
        i = perm[a0 + p];
        j = perm[b0 + pm];
    } else {
        i = perm[a0 + pm];
        j = perm[b0 + p];
    }
}

// Energy pairs of one species forward (Algorithm 1, final loop), by one warp, 32 pairs of a pass at a time: caps fE K, a
// prefix sum over them, capped pairs take their cap and the crossing pair the remainder of |D|. Every pair that
// absorbed energy is taped from entry e0 on, in order; returns their number. D = 0: Delta E_s vanishes here (exactly,
// or as rounding noise), so the step applies no pair; but it moves at first order with v and w, and then the first
// pair of the order absorbs it as the crossing pair: that pair is taped with U = 0. done: D was absorbed.
__device__ int energy_forward(const StepArgs& A, const Slab& sl, const Work& wk, int N, int s0, int ns, double msd,
                              double D, int e0, bool& done)
{
    const int lane = threadIdx.x & 31;
    const bool none = D == 0.0;
    const double sgn = D > 0.0 ? 1.0 : -1.0;
    double Dabs = fabs(D);
    int used = 0;
    done = none;
    const int passes = none ? 1 : A.max_corr_passes;
    bool stop = false;
    static_assert(kWarps == 4, "the prefix sums below are those of the step kernel's four warps");
    for (int pass = 0; pass < passes && !stop; ++pass) {
        const int o = pass & 1, np = (ns - o) / 2;
        double carry = 0.0;
        // Chunks of kThreads pairs as in the step kernel, 32 at a time. Its prefix sums: within a warp, then over its warps'
        // totals, offsets t0, t1 + t0, (t2 + t1) + t0 and total (t3 + t2) + (t1 + t0), then the chunks before.
        for (int chunk = 0; chunk < np && !stop; chunk += kThreads) {
            double t0 = 0.0, t1 = 0.0, t2 = 0.0, t3 = 0.0;
            for (int grp = 0; grp < kWarps && chunk + 32 * grp < np && !stop; ++grp) {
                const int m = chunk + 32 * grp + lane;
                int i = 0, j = 0;
                double v1[3], v2[3], m1 = 1.0, m2 = 1.0, K = 0.0;
                if (m < np) {
                    i = wk.rho[s0 + o + 2 * m];
                    j = wk.rho[s0 + o + 2 * m + 1];
                    ld3(wk.v, N, i, v1);
                    ld3(wk.v, N, j, v2);
                    m1 = msd * wk.w[i];
                    m2 = msd * wk.w[j];
                    K = pair_kecm<double, false>(A.c, m1, m2, v1, v2);
                }
                const bool ok = K > 0.0;
                bool take;
                double U = 0.0, capE = 0.0;
                if (none) {
                    const unsigned b = __ballot_sync(0xffffffffu, ok);
                    take = ok && lane == __ffs(b) - 1;
                    stop = b != 0;
                } else {
                    capE = ok ? A.fE * K : 0.0;
                    double inc = capE;
#pragma unroll
                    for (int q = 1; q < 32; q <<= 1) {
                        const double y = __shfl_up_sync(0xffffffffu, inc, q);
                        if (lane >= q) inc += y;
                    }
                    const double off = grp == 0 ? 0.0 : (grp == 1 ? t0 : (grp == 2 ? t1 + t0 : (t2 + t1) + t0));
                    double excl = __shfl_up_sync(0xffffffffu, inc, 1);
                    excl = (off + (lane ? excl : 0.0)) + carry;
                    take = ok && excl < Dabs;
                    const double rem = Dabs - excl;
                    U = sgn * (rem < capE ? rem : capE);
                    const double t = __shfl_sync(0xffffffffu, inc, 31);
                    if (grp == 0) t0 = t;
                    else if (grp == 1) t1 = t;
                    else if (grp == 2) t2 = t;
                    else t3 = t;
                    // the step kernel's shortcut: the first 32 pairs absorb all of it
                    if (pass == 0 && chunk == 0 && grp == 0) stop = done = t >= Dabs;
                }
                const unsigned b = __ballot_sync(0xffffffffu, take);
                if (take) {
                    const int e = e0 + used + __popc(b & ((1u << lane) - 1u));
                    if (e < sl.E) {
                        for (int k = 0; k < 3; ++k) {
                            sl.ev[k * sl.E + e] = v1[k];
                            sl.ev[(3 + k) * sl.E + e] = v2[k];
                        }
                        sl.ei[e] = i;
                        sl.ej[e] = j;
                        sl.eU[e] = U;
                        sl.eK[e] = K;
                        sl.ecap[e] = 2 * pass + (!none && fabs(U) == capE);
                    } else if (!none) {
                        latch(A.status, kErrTooLarge);
                    }
                    if (!none) {
                        energy_pair<double, false>(A.c, m1, m2, K, v1, v2, U);
                        st3(wk.v, N, i, v1);
                        st3(wk.v, N, j, v2);
                    }
                }
                used += __popc(b);
                __syncwarp();
            }
            carry += (t3 + t2) + (t1 + t0);
            if (!none && carry >= Dabs) stop = done = true;
        }
        Dabs -= carry;
    }
    return used;
}

// The same pairs backwards, by one warp: from the last entry, up to 32 entries of one pass at a time (disjoint particles).
// Adds to the gradients at the pairs' particles and weights; returns dL/dD of the species.
__device__ double energy_reverse(const StepArgs& A, const Slab& sl, const Work& wk, int N, int e0, int cnt, double msd,
                                 double D)
{
    const int lane = threadIdx.x & 31;
    const double sgn = D > 0.0 ? 1.0 : -1.0;
    double gUc = 0.0, gD = 0.0;
    for (int left = cnt; left > 0;) {
        const int k = e0 + left - 1 - lane;  // lane 0 takes the last entry
        const int cap = lane < left ? sl.ecap[k] : -2;
        const bool mine = (cap >> 1) == (__shfl_sync(0xffffffffu, cap, 0) >> 1);
        const int n = __popc(__ballot_sync(0xffffffffu, mine));  // a pass's entries are consecutive
        int i = 0, j = 0;
        double vr[3], g1[3], g2[3], h[3], m1 = 1.0, m2 = 1.0, K = 1.0, x = 0.0, gg = 1.0, ggm1 = 0.0, g1vr = 0.0,
                                                                  g2vr = 0.0, vr2 = 0.0;
        if (mine) {
            i = sl.ei[k];
            j = sl.ej[k];
            ld3(wk.v, N, i, g1);
            ld3(wk.v, N, j, g2);
            m1 = msd * wk.w[i];
            m2 = msd * wk.w[j];
            K = sl.eK[k];
            x = sl.eU[k] / K;
            gg = sqrt(1.0 - x);
            const double rM = 1.0 / (m1 + m2);
            for (int d = 0; d < 3; ++d) {
                vr[d] = sl.ev[d * sl.E + k] - sl.ev[(3 + d) * sl.E + k];
                h[d] = (m2 * g1[d] - m1 * g2[d]) * rM;
                ggm1 += h[d] * vr[d];
                g1vr += g1[d] * vr[d];
                g2vr += g2[d] * vr[d];
                vr2 += vr[d] * vr[d];
            }
        }
        // the crossing pair: U = D - (earlier U); g - 1 depends on U and K. It is the last entry, if there is one.
        const bool crossing = mine && !(cap & 1);
        const double gU = crossing ? -ggm1 / (2.0 * gg * K) : 0.0;
        if (left == cnt) {
            gD = __shfl_sync(0xffffffffu, gU, 0);
            gUc = gD;
        }
        if (mine) {
            const double gm1 = -x / (1.0 + gg), rM = 1.0 / (m1 + m2);
            const double gc1 = gm1 * g1vr, gc2 = -gm1 * g2vr;
            // a capped pair has U = sign(D) fE K, so U/K is fixed; its K still feeds the crossing pair's U
            const double gK = crossing ? -gU * x : -gUc * sgn * A.fE;
            const double mu = m1 * m2 * rM, gmu = gK * 0.5 * vr2, rM2 = rM * rM;
            const double gm1m = (gmu * m2 - gc1 + gc2) * m2 * rM2;
            const double gm2m = (gmu * m1 + gc1 - gc2) * m1 * rM2;
            wk.gwl[i] += msd * gm1m;
            wk.gwl[j] += msd * gm2m;
            for (int d = 0; d < 3; ++d) {
                const double gv = gm1 * h[d] + gK * mu * vr[d];
                g1[d] += gv;
                g2[d] -= gv;
            }
            st3(wk.v, N, i, g1);
            st3(wk.v, N, j, g2);
        }
        left -= n;
        __syncwarp();
    }
    return gD;
}

__global__ void __launch_bounds__(kThreads, kAdjCtasPerSm) k_adjoint(const __grid_constant__ AdjArgs G)
{
    extern __shared__ __align__(16) char dyn[];
    __shared__ AdjShared sh;
    const StepArgs& A = G.a;
    const InterConst& ic = A.ic[0];
    const int S = A.S;
    const bool intra = ic.a == ic.b;
    const double* wg = A.w;
    const double* gvx = reinterpret_cast<const double*>(A.vx);
    const double* gvy = reinterpret_cast<const double*>(A.vy);
    const double* gvz = reinterpret_cast<const double*>(A.vz);
    const uint32_t ictr = (uint32_t)A.inter_base;
    const bool keep = G.gx || G.tape == 1;  // a forward that is neither reversed nor recorded needs no tape
    for (int c = blockIdx.x; c < A.n_cells; c += gridDim.x) {
        const Slab sl = make_slab(G.slab + (size_t)(G.tape ? c : (int)blockIdx.x) * (size_t)G.slab_stride, G.max_cell,
                                  G.max_epairs);
        const Work wk = make_work(G.on_chip ? dyn : sl.work, G.max_cell);
        const int64_t cs = A.offsets[(int64_t)c * S];
        const int n = (int)(A.offsets[(int64_t)(c + 1) * S] - cs);
        const int N = sl.n;
        if (n > N) {
            if (threadIdx.x == 0) latch(A.status, kErrBounds);
            continue;
        }
        if ((int)threadIdx.x <= S) sh.off[threadIdx.x] = (int)(A.offsets[(int64_t)c * S + threadIdx.x] - cs);
        for (int i = threadIdx.x; i < n; i += kThreads) {
            wk.w[i] = wg[cs + i];
            if (G.tape != 2) {  // a replaying call finds the state before the interaction in the tape
                const double x[3] = {gvx[cs + i], gvy[cs + i], gvz[cs + i]};
                st3(wk.v, N, i, x);
                st3(sl.vb, N, i, x);
            }
        }
        __syncthreads();
        const int a0 = sh.off[ic.a], na = sh.off[ic.a + 1] - a0;
        const int b0 = sh.off[ic.b], nb = sh.off[ic.b + 1] - b0;
        const bool active = intra ? (na >= 2) : (na > 0 && nb > 0);
        const int nside = intra ? 1 : 2;
        if (active && G.tape == 2) {
            // ---- replay: the forward's per-cell scalars from the tape
            if (threadIdx.x == 0) {
                const TapeHead& h = *sl.head;
                sh.fail = h.fail;
                for (int k = 0; k < 2; ++k) {
                    sh.ne[k] = h.ne[k];
                    sh.e0[k] = h.e0[k];
                    sh.zeroed[k] = h.zeroed[k];
                    sh.Es[k] = h.Es[k];
                    sh.W1[k] = h.W1[k];
                    sh.D[k] = h.D[k];
                }
                for (int k = 0; k < 3; ++k) {
                    sh.B[k] = h.B[k];
                    sh.S[k] = h.S[k];
                }
                sh.Sw = h.Sw;
                sh.dE = h.dE;
            }
            __syncthreads();
        } else if (active) {
            // ---- forward: permutations
            cta_permutations(A.rng, A.rng.step, wk.keys, wk.cnt, wk.perm, sh.iscan, c, ictr, nside, a0, na, b0, nb);
            // ---- forward: scatter pairs in round order, inputs taped
            const int npairs = intra ? ((na & 1) ? (na + 3) / 2 : na / 2) : (na > nb ? na : nb);
            const int nmin = intra ? na - 1 : (na < nb ? na : nb);
            const int lead = (intra && (na & 1)) ? 3 : 0;
            const int round = intra ? npairs : nmin;
            for (int r0 = 0; r0 < npairs; r0 += round) {
                const int r1 = r0 + round < npairs ? r0 + round : npairs;
                int p = (lead && threadIdx.x == 0) ? 0 : r0 + lead + (int)threadIdx.x;
                while (p < r1) {
                    int i, j;
                    bool trip;
                    pair_of(wk.perm, intra, na, nb, a0, b0, p, p - r0, i, j, trip);
                    double vi[3], vj[3];
                    ld3(wk.v, N, i, vi);
                    ld3(wk.v, N, j, vj);
                    const uint4 rr = draw(A.rng, (uint32_t)p, (uint32_t)c, ictr, kTagScat);
                    const int flags = pair_forward(A, ic, vi, vj, wk.w[i], wk.w[j], nmin, trip, rr,
                                                   keep ? sl.pv + p : nullptr, (size_t)N);
                    if (keep) {
                        sl.pi[p] = i | flags;
                        sl.pj[p] = j;
                    }
                    st3(wk.v, N, i, vi);
                    st3(wk.v, N, j, vj);
                    p = (p + 1 < lead) ? p + 1 : (p < lead ? lead + (int)threadIdx.x : p + kThreads);
                }
                __syncthreads();
            }
            // ---- forward: moment correction
            if (A.correct) {
                // the sums and coefficients of the step kernel, term for term and in its order
                const double ms[2] = {A.m[ic.a], A.m[ic.b]};
                {
                    Acc<double> mom[6], wsum[4];
                    for (int k = 0; k < 6; ++k) mom[k] = Acc<double>::zero();
                    for (int k = 0; k < 4; ++k) wsum[k] = Acc<double>::zero();
                    for (int side = 0; side < nside; ++side) {
                        const int s0 = side ? b0 : a0, ns = side ? nb : na;
                        for (int q = threadIdx.x; q < ns; q += kThreads) {
                            const int i = s0 + q;
                            const double w = wk.w[i];
                            for (int k = 0; k < 3; ++k) mom[3 * side + k].add(w * (wk.v[k * N + i] - sl.vb[k * N + i]));
                            wsum[2 * side].add(w);
                            wsum[2 * side + 1].add(w * w);
                        }
                    }
                    block_sum<double, 4>(wsum, accp(sh.red_raw), accp(sh.red));
                    if (threadIdx.x == 0) {
                        const Acc<double>* r = accp(sh.red);
                        sh.W1[0] = r[0].x;
                        sh.W1[1] = r[2].x;
                        sh.Sw = mass_sum(ms[0], r[1].x, ms[1], r[3].x, intra);
                    }
                    __syncthreads();
                    block_sum<double, 6>(mom, accp(sh.red_raw), accp(sh.red));
                    if (threadIdx.x == 0) {
                        const Acc<double>* r = accp(sh.red);
                        for (int k = 0; k < 3; ++k) {
                            sh.S[k] = mass_sum(ms[0], r[k].x, ms[1], r[3 + k].x, intra);
                            sh.B[k] = sh.S[k] / sh.Sw;
                        }
                    }
                    __syncthreads();
                }
                {
                    Acc<double> acc[4];
                    for (int k = 0; k < 4; ++k) acc[k] = Acc<double>::zero();
                    for (int side = 0; side < nside; ++side) {
                        const int s0 = side ? b0 : a0, ns = side ? nb : na;
                        for (int q = threadIdx.x; q < ns; q += kThreads) {
                            const int i = s0 + q;
                            const double w = wk.w[i];
                            double dd = 0.0, v2 = 0.0;
                            for (int k = 0; k < 3; ++k) {
                                const double x = wk.v[k * N + i] - sh.B[k] * w, y = sl.vb[k * N + i];
                                wk.v[k * N + i] = x;
                                if (keep) sl.vm[k * N + i] = x;
                                dd += (x - y) * (x + y);
                                v2 += x * x;
                            }
                            acc[2 * side].add(0.5 * w * dd);
                            acc[2 * side + 1].add(0.5 * w * v2);
                        }
                    }
                    block_sum<double, 4>(acc, accp(sh.red_raw), accp(sh.red));
                    if (threadIdx.x == 0) {
                        const Acc<double>* r = accp(sh.red);
                        const double dE = mass_sum(ms[0], r[0].x, ms[1], r[2].x, intra);
                        sh.dE = dE;
                        sh.Es[0] = __dmul_rn(ms[0], r[1].x);
                        sh.Es[1] = intra ? 0.0 : __dmul_rn(ms[1], r[3].x);
                        double D0, D1;
                        const int fail = split64(intra, na, nb, split_weight64(sh.W1[0], na, sh.Es[0]),
                                                 split_weight64(sh.W1[1], nb, sh.Es[1]), dE, D0, D1);
                        sh.zeroed[0] = fabs(D0) <= 0x1p-47 * sh.Es[0];
                        sh.zeroed[1] = fabs(D1) <= 0x1p-47 * (intra ? 0.0 : sh.Es[1]);
                        sh.D[0] = sh.zeroed[0] ? 0.0 : D0;
                        sh.D[1] = sh.zeroed[1] ? 0.0 : D1;
                        sh.fail = sh.fail0 = fail;
                    }
                    __syncthreads();
                }
                // energy-pair order of each side: the permutation, stably sorted by descending weight (optional)
                for (int side = 0; side < nside; ++side) {
                    const int s0 = side ? b0 : a0, ns = side ? nb : na;
                    if (!A.sort_by_weight) {
                        for (int r = threadIdx.x; r < ns; r += kThreads) wk.rho[s0 + r] = wk.perm[s0 + r];
                        continue;
                    }
                    for (int r = threadIdx.x; r < ns; r += kThreads)
                        wk.keys[s0 + r] = weight_key(wk.w[wk.perm[s0 + r]], (uint32_t)r);
                }
                __syncthreads();
                if (A.sort_by_weight) {
                    for (int side = 0; side < nside; ++side) block_sort_u64(wk.keys + (side ? b0 : a0), side ? nb : na);
                    for (int side = 0; side < nside; ++side) {
                        const int s0 = side ? b0 : a0, ns = side ? nb : na;
                        for (int r = threadIdx.x; r < ns; r += kThreads)
                            wk.rho[s0 + r] = wk.perm[s0 + (int)(wk.keys[s0 + r] & kPermMask)];
                    }
                    __syncthreads();
                }
                // energy pairs, one warp per side: at once under the rollback policy (a failure undoes both), else
                // species b only if species a did not fail. Side b's tape starts after the most that side a can need.
                const int turns = A.fail_policy == 0 ? 1 : nside;
                const int passes = A.max_corr_passes > 0 ? A.max_corr_passes : 1;
                for (int turn = 0; turn < turns; ++turn) {
                    const int side = threadIdx.x >> 5;
                    if (side < nside && (turns == 1 || side == turn)) {
                        const int e0 = side ? passes * (na / 2) : 0;
                        int used = 0;
                        bool done = true;
                        if (!(turns == 1 ? sh.fail0 : sh.fail))
                            used = energy_forward(A, sl, wk, N, side ? b0 : a0, side ? nb : na, ms[side], sh.D[side], e0,
                                                  done);
                        if ((threadIdx.x & 31) == 0) {
                            sh.e0[side] = e0;
                            sh.ne[side] = used;
                            if (!done) sh.fail = 1;
                        }
                    }
                    __syncthreads();
                }
                if (sh.fail && A.fail_policy == 0) {
                    for (int side = 0; side < nside; ++side) {
                        const int s0 = side ? b0 : a0, ns = side ? nb : na;
                        for (int q = threadIdx.x; q < ns; q += kThreads) {
                            double x[3];
                            ld3(sl.vb, N, s0 + q, x);
                            st3(wk.v, N, s0 + q, x);
                        }
                    }
                }
                if (sh.fail && A.fail_policy == 2 && threadIdx.x == 0) latch(A.status, kErrCorrectionFailed);
                __syncthreads();
            }
            if (G.tape == 1 && threadIdx.x == 0) {  // record: keep the per-cell scalars with the tape
                TapeHead& h = *sl.head;
                h.fail = A.correct ? sh.fail : 0;
                for (int k = 0; k < 2; ++k) {
                    h.ne[k] = sh.ne[k];
                    h.e0[k] = sh.e0[k];
                    h.zeroed[k] = sh.zeroed[k];
                    h.Es[k] = sh.Es[k];
                    h.W1[k] = sh.W1[k];
                    h.D[k] = sh.D[k];
                }
                for (int k = 0; k < 3; ++k) {
                    h.B[k] = sh.B[k];
                    h.S[k] = sh.S[k];
                }
                h.Sw = sh.Sw;
                h.dE = sh.dE;
            }
        }
        // ---- forward output
        if (G.ox) {
            for (int i = threadIdx.x; i < n; i += kThreads) {
                G.ox[cs + i] = wk.v[i];
                G.oy[cs + i] = wk.v[N + i];
                G.oz[cs + i] = wk.v[2 * N + i];
            }
        }
        // ---- reverse
        if (G.gx && active && !(A.correct && sh.fail && A.fail_policy == 0)) {
            __syncthreads();  // the forward's working arrays are read no more
            for (int i = threadIdx.x; i < n; i += kThreads) {
                const double x[3] = {G.gx[cs + i], G.gy[cs + i], G.gz[cs + i]};
                st3(wk.v, N, i, x);
                const double z[3] = {0.0, 0.0, 0.0};
                st3(wk.gb, N, i, z);
                wk.gwl[i] = 0.0;
            }
            __syncthreads();
            if (A.correct) {
                const double ms[2] = {A.m[ic.a], A.m[ic.b]};
                // energy pairs backwards, one warp per side (their particles are disjoint)
                {
                    const int side = threadIdx.x >> 5;
                    if (side < nside) {
                        const int cnt = sh.ne[side] < sl.E - sh.e0[side] ? sh.ne[side] : sl.E - sh.e0[side];
                        const double gD = energy_reverse(A, sl, wk, N, sh.e0[side], cnt, ms[side], sh.D[side]);
                        if ((threadIdx.x & 31) == 0) sh.gD[side] = gD;
                    }
                }
                __syncthreads();
                if (threadIdx.x == 0) {
                    // Delta E split backwards
                    double gdE = 0.0, gE0 = 0.0, gE1 = 0.0, gW0 = 0.0, gW1 = 0.0;
                    const double g0 = sh.gD[0];
                    const double g1 = intra ? 0.0 : sh.gD[1];
                    if (intra) {
                        gdE = g0;
                    } else {
                        const bool c0 = na >= 2, c1 = nb >= 2;
                        if (c0 && c1) {
                            const double wa = sh.W1[0] / (double)na * sh.Es[0];
                            const double wb = sh.W1[1] / (double)nb * sh.Es[1];
                            const double den = wa + wb;
                            if (den > 0.0) {
                                const double f = wa / den;
                                gdE = g1 + (g0 - g1) * f;
                                const double gf = (g0 - g1) * sh.dE;
                                const double gwa = gf * wb / (den * den), gwb = -gf * wa / (den * den);
                                gW0 = gwa * sh.Es[0] / (double)na;
                                gE0 = gwa * sh.W1[0] / (double)na;
                                gW1 = gwb * sh.Es[1] / (double)nb;
                                gE1 = gwb * sh.W1[1] / (double)nb;
                            }
                        } else if (c0) {
                            gdE = g0;
                        } else if (c1) {
                            gdE = g1;
                        }
                    }
                    sh.gdE = gdE;
                    sh.gEs[0] = gE0;
                    sh.gEs[1] = gE1;
                    sh.gW1[0] = gW0;
                    sh.gW1[1] = gW1;
                }
                __syncthreads();
                // energy sums and the momentum shift backwards: g at v_pm, then g_B = -sum w g_vpm
                {
                    Acc<double> acc[3];
                    for (int k = 0; k < 3; ++k) acc[k] = Acc<double>::zero();
                    for (int side = 0; side < nside; ++side) {
                        const int s0 = side ? b0 : a0, ns = side ? nb : na;
                        const double msd = ms[side];
                        for (int q = threadIdx.x; q < ns; q += kThreads) {
                            const int i = s0 + q;
                            const double w = wk.w[i], mp = msd * w;
                            double gm[3], xm[3], xb[3];
                            ld3(wk.v, N, i, gm);
                            ld3(sl.vm, N, i, xm);
                            ld3(sl.vb, N, i, xb);
                            const double gE = sh.gEs[side];
                            double xm2 = 0.0, xb2 = 0.0, gwd = 0.0;
                            for (int d = 0; d < 3; ++d) {
                                gm[d] += (sh.gdE + gE) * mp * xm[d];
                                wk.gb[d * N + i] -= sh.gdE * mp * xb[d];
                                xm2 += xm[d] * xm[d];
                                xb2 += xb[d] * xb[d];
                            }
                            gwd += sh.gdE * 0.5 * msd * (xm2 - xb2) + gE * 0.5 * msd * xm2 + sh.gW1[side];
                            for (int d = 0; d < 3; ++d) {
                                acc[d].add(-w * gm[d]);
                                gwd -= sh.B[d] * gm[d];
                            }
                            wk.gwl[i] += gwd;
                            st3(wk.v, N, i, gm);
                        }
                    }
                    block_sum<double, 3>(acc, accp(sh.red_raw), accp(sh.red));
                    if (threadIdx.x == 0) {
                        const Acc<double>* r = accp(sh.red);
                        double gSw = 0.0;
                        for (int d = 0; d < 3; ++d) {
                            sh.gS[d] = r[d].x / sh.Sw;
                            gSw -= r[d].x * sh.B[d] / sh.Sw;
                        }
                        sh.gSw = gSw;
                    }
                    __syncthreads();
                }
                // B = S / Sw, S = sum m w (v_ps - v_bs), Sw = sum m w^2 backwards
                for (int side = 0; side < nside; ++side) {
                    const int s0 = side ? b0 : a0, ns = side ? nb : na;
                    const double msd = ms[side];
                    for (int q = threadIdx.x; q < ns; q += kThreads) {
                        const int i = s0 + q;
                        const double w = wk.w[i], mp = msd * w;
                        double gwd = 2.0 * mp * sh.gSw;
                        for (int d = 0; d < 3; ++d) {
                            wk.v[d * N + i] += mp * sh.gS[d];
                            wk.gb[d * N + i] -= mp * sh.gS[d];
                            gwd += msd * ((sl.vm[d * N + i] - sl.vb[d * N + i]) + sh.B[d] * w) * sh.gS[d];  // v_ps = v_pm + B w
                        }
                        wk.gwl[i] += gwd;
                    }
                }
                __syncthreads();
            }
            // scatter pairs backwards: rounds in reverse, the odd triplet in reverse by thread 0
            double glnl = 0.0;  // lnL dL/dlnL
            {
                const int npairs = intra ? ((na & 1) ? (na + 3) / 2 : na / 2) : (na > nb ? na : nb);
                const int nmin = intra ? na - 1 : (na < nb ? na : nb);
                const int lead = (intra && (na & 1)) ? 3 : 0;
                const int round = intra ? npairs : nmin;
                const int nround = (npairs + round - 1) / round;
                for (int rr = nround - 1; rr >= 0; --rr) {
                    const int r0 = rr * round;
                    const int r1 = r0 + round < npairs ? r0 + round : npairs;
                    // the triplet (0, 1, 2) shares particles: thread 0 undoes it in reverse; the other pairs of the round
                    // are disjoint from it and from each other
                    auto undo = [&](int p) {
                        const int f = sl.pi[p], i = f & kPairIndex, j = sl.pj[p];
                        double g1[3], g2[3];
                        ld3(wk.v, N, i, g1);
                        ld3(wk.v, N, j, g2);
                        double gwi = 0.0, gwj = 0.0;
                        glnl += pair_reverse(ic, G.lnL, sl.pv + p, N, wk.w[i], wk.w[j], f, g1, g2, gwi, gwj);
                        st3(wk.v, N, i, g1);
                        st3(wk.v, N, j, g2);
                        wk.gwl[i] += gwi;
                        wk.gwl[j] += gwj;
                    };
                    if (lead && threadIdx.x == 0)
                        for (int p = lead - 1; p >= 0; --p) undo(p);
                    for (int p = r0 + lead + (int)threadIdx.x; p < r1; p += kThreads) undo(p);
                    __syncthreads();
                }
            }
            // dL/dv_before = scatter path + direct correction path; dL/dw, dL/dlnL accumulated
            for (int side = 0; side < nside; ++side) {
                const int s0 = side ? b0 : a0, ns = side ? nb : na;
                for (int q = threadIdx.x; q < ns; q += kThreads) {
                    const int i = s0 + q;
                    G.gx[cs + i] = wk.v[i] + wk.gb[i];
                    G.gy[cs + i] = wk.v[N + i] + wk.gb[N + i];
                    G.gz[cs + i] = wk.v[2 * N + i] + wk.gb[2 * N + i];
                    if (G.gw) G.gw[cs + i] += wk.gwl[i];
                }
            }
            {
                Acc<double> acc[1] = {Acc<double>{glnl}};
                block_sum<double, 1>(acc, accp(sh.red_raw), accp(sh.red));
                if (threadIdx.x == 0 && G.glnL) atomicAdd(G.glnL, accp(sh.red)[0].x != 0.0 ? accp(sh.red)[0].x / G.lnL : 0.0);
            }
        }
        __syncthreads();
    }
}

}  // namespace

size_t adjoint_slab_bytes(int32_t max_cell, int32_t max_epairs, bool on_chip)
{
    return (slab_bytes(max_cell, max_epairs, on_chip) + 255) & ~(size_t)255;
}

size_t adjoint_work_bytes(int32_t max_cell) { return kWorkBytesPerParticle * (size_t)max_cell; }

size_t adjoint_static_smem()
{
    cudaFuncAttributes fa;
    return cudaFuncGetAttributes(&fa, k_adjoint) == cudaSuccess ? fa.sharedSizeBytes : 16384;
}

cudaError_t set_adjoint_smem_limit(size_t smem)
{
    return cudaFuncSetAttribute(k_adjoint, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

int adjoint_ctas_per_sm() { return kAdjCtasPerSm; }

cudaError_t launch_adjoint(const StepArgs& a, double lnL, double* ox, double* oy, double* oz, double* gx, double* gy,
                           double* gz, double* gw, double* glnL, char* slab, int32_t max_cell, int32_t max_epairs,
                           int32_t tape, bool on_chip, int grid, cudaStream_t st)
{
    AdjArgs g;
    g.a = a;
    g.lnL = lnL;
    g.ox = ox;
    g.oy = oy;
    g.oz = oz;
    g.gx = gx;
    g.gy = gy;
    g.gz = gz;
    g.gw = gw;
    g.glnL = glnL;
    g.slab = slab;
    g.slab_stride = (int64_t)adjoint_slab_bytes(max_cell, max_epairs, on_chip);
    g.max_cell = max_cell;
    g.max_epairs = max_epairs;
    g.tape = tape;
    g.on_chip = on_chip;
    const size_t smem = on_chip ? adjoint_work_bytes(max_cell) : 0;
    k_adjoint<<<grid, kThreads, smem, st>>>(g);
    return cudaGetLastError();
}

}  // namespace mcc
