// hfs_schedule.cuh -- the FP64 stage flows and phase records as device
// functions (the formulas are described in hfs_schedule.cu), for the schedule
// kernels and for the step kernel of few instances, which makes its own.
#pragma once

#include "hfs_internal.cuh"
#include "hfs_law.cuh"
#include "hfs_sched.h"

namespace hfs {

// C = cos(sqrt(w) t), S = sin(sqrt(w) t)/sqrt(w), OMC = 1 - C, continued to w <= 0
struct CS {
    double C, S, OMC;
};
__device__ inline CS cs_of(double w, double t)
{
    CS r;
    const double z = w * t * t;  // theta^2, negative for w < 0
    if (fabs(z) <= 1e-3) {
        // the same series to z^3: the first omitted terms, z^4/10! and z^4/9!,
        // are below 3e-18 of the sums
        const double c = fma(fma(fma(-z, 1.0 / 40320.0, 1.0 / 720.0), -z, 1.0 / 24.0), -z, 0.5);
        const double sv = fma(fma(fma(-z, 1.0 / 5040.0, 1.0 / 120.0), -z, 1.0 / 6.0), -z, 1.0);
        r.OMC = z * c;
        r.C = 1.0 - r.OMC;
        r.S = t * sv;
        return r;
    }
    if (fabs(z) <= 0.25) {
        // Power series of the entire functions in z = w t^2 (Taylor series of
        // cos and sin / theta), eight terms: truncation below 1e-18.  No square
        // root, no division, and w <= 0 needs no separate branch.
        double c = 1.0 / 20922789888000.0, s = 1.0 / 1307674368000.0;
        c = fma(c, -z, 1.0 / 87178291200.0);
        c = fma(c, -z, 1.0 / 479001600.0);
        c = fma(c, -z, 1.0 / 3628800.0);
        c = fma(c, -z, 1.0 / 40320.0);
        c = fma(c, -z, 1.0 / 720.0);
        c = fma(c, -z, 1.0 / 24.0);
        c = fma(c, -z, 1.0 / 2.0);  // (1 - C)/z
        s = fma(s, -z, 1.0 / 6227020800.0);
        s = fma(s, -z, 1.0 / 39916800.0);
        s = fma(s, -z, 1.0 / 362880.0);
        s = fma(s, -z, 1.0 / 5040.0);
        s = fma(s, -z, 1.0 / 120.0);
        s = fma(s, -z, 1.0 / 6.0);
        s = fma(s, -z, 1.0);  // S / t
        r.OMC = z * c;
        r.C = 1.0 - r.OMC;
        r.S = t * s;
        return r;
    }
    if (w > 0.0) {
        const double q = sqrt(w);
        double sh, ch;
        sincos(0.5 * q * t, &sh, &ch);
        r.C = 1.0 - 2.0 * sh * sh;
        r.OMC = 2.0 * sh * sh;
        r.S = 2.0 * sh * ch / q;
    } else {
        const double q = sqrt(-w);
        const double sh = sinh(0.5 * q * t), ch = cosh(0.5 * q * t);
        r.C = 1.0 + 2.0 * sh * sh;
        r.OMC = -2.0 * sh * sh;
        r.S = 2.0 * sh * ch / q;
    }
    return r;
}

// Theorem 2 for the product of two half steps (R applied first), mu = 1
__device__ inline void fge_thm2(double wl, double wr, double s, double &f, double &g, double &e)
{
    const CS L = cs_of(wl, 0.5 * s), Rr = cs_of(wr, 0.5 * s);
    g = L.S * Rr.C + L.C * Rr.S;
    const double omcc = L.OMC + L.C * Rr.OMC;  // 1 - C_L C_R
    const double ss = L.S * Rr.S;
    const double ig = 1.0 / g;
    f = (omcc + wl * ss) * ig;
    e = (omcc + wr * ss) * ig;
}

// Theorem 1 for exp(-i s/2 (al x^2 + be (xp+px) + ga p^2))
__device__ inline void fge_thm1(double al, double be, double ga, double s, double &f, double &g, double &e)
{
    const CS r = cs_of(al * ga - be * be, s);
    g = ga * r.S;
    const double ig = 1.0 / g;
    f = (r.OMC + be * r.S) * ig;
    e = (r.OMC - be * r.S) * ig;
}

constexpr double kR3 = 0.28867513459481288225;   // sqrt(3)/6
constexpr double kR15 = 0.38729833462074168852;  // sqrt(15)/10

// The trap's shape factors S (omega^2 = omega0^2 S) of one stage over
// [tau, tau + s] at the nodes its flow reads: the stage start (Lemma 2), the
// two Gauss nodes (Magnus-4), the three Gauss nodes (Magnus-6).
struct NodeS {
    double s[3];
};

template <int FLOW, int LAW> __device__ __forceinline__ NodeS stage_nodes(const DevInst &p, double tau, double s)
{
    NodeS r{};
    if constexpr (FLOW == HFS_FLOW_LEMMA2) {
        r.s[0] = law_factor<LAW>(p, tau);
    } else if constexpr (FLOW == HFS_FLOW_CF4) {
        law_factor_pair<LAW>(p, tau + 0.5 * s, kR3 * s, r.s[0], r.s[1]);
    } else {
        law_factor_pair<LAW>(p, tau + 0.5 * s, kR15 * s, r.s[0], r.s[2]);
        r.s[1] = law_factor<LAW>(p, tau + 0.5 * s);
    }
    return r;
}

// (f, g, e) of one stage on axis `axis` from the shape factors at its nodes.
// FLOW (and LAW, SHARED below) are template parameters: with a run-time flow
// the compiler evaluated all three branches and kept one result (3.6x the
// FP64 work).
template <int FLOW>
__device__ void stage_fge(const DevInst &p, int dim, int axis, const NodeS &ns, double s, double &f, double &g,
                          double &e)
{
    const double c = (dim == 1) ? 1.0 : p.axis_scale[axis];
    const double k = c * c * (p.w0 * p.w0);  // omega^2 = k S
    if constexpr (FLOW == HFS_FLOW_LEMMA2) {
        const double om = sqrt(k * ns.s[0]);
        double sh, ch;
        sincos(0.5 * om * s, &sh, &ch);
        g = 2.0 * sh * ch / om;
        f = om * sh / ch;
        e = f;
    } else if constexpr (FLOW == HFS_FLOW_CF4) {
        const double al = 0.5 - 2.0 * kR3;  // 1/2 - 1/sqrt(3)
        const double be = 1.0 - al;
        const double w1 = k * ns.s[0], w2 = k * ns.s[1];
        fge_thm2(al * w1 + be * w2, be * w1 + al * w2, s, f, g, e);
    } else {
        const double w1 = k * ns.s[0], w2 = k * ns.s[1], w3 = k * ns.s[2];
        const double s2 = s * s;
        const double avg = 5.0 * w1 + 8.0 * w2 + 5.0 * w3;
        const double al = avg / 18.0 + s2 / 486.0 * (4.25 * (w1 * w1 + w3 * w3) + 8.0 * w2 * w2 + w1 * w2 +
                                                     w2 * w3 - 18.5 * w1 * w3);
        const double be = s * 1.29099444873580562839 * (w3 - w1) * (1.0 / 12.0 + s2 / 3240.0 * avg);  // sqrt(5/3)
        const double ga = 1.0 + s2 / 54.0 * (w1 - 2.0 * w2 + w3);
        fge_thm1(al, be, ga, s, f, g, e);
    }
    // mass: the mu-problem is the mu = 1 problem conjugated by diag(1, mu)
    if (p.mu != 1.0) {
        f *= p.mu;
        e *= p.mu;
        g /= p.mu;
    }
}

// kick coefficient kappa, B sum and drift g of sub-stage j on axis d
template <int SPLIT>
__device__ void merged_coeffs(const DevInst &p, int dim, int d, const SchedConst &sc, double t0, int j, int nstage,
                              const StageFGE *__restrict__ fge_i, double &kappa, double &bs, double &g)
{
    const int mm = sc.m;
    const int r = j % mm;
    if (r == 0) bs = (j > 0 ? sc.b[mm] : 0.0) + (j < nstage ? sc.b[0] : 0.0);
    else bs = sc.b[r];
    if constexpr (SPLIT == HFS_SPLIT_HO) {
        kappa = 0.0;
        if (j >= 1) kappa += fge_i[(j - 1) * dim + d].f;
        if (j < nstage) kappa += fge_i[j * dim + d].e;
        g = (j < nstage) ? fge_i[j * dim + d].g : 0.0;
    } else {
        // F split: B carries mu omega^2(tau_j) x^2/2 with the time frozen at the stage boundary
        const double tau = t0 + (double)(j / mm) * sc.h + sc.h * sc.cuma[r];
        kappa = bs * sc.h * p.mu * axis_omega2(p, dim, d, tau);
        g = (j < nstage) ? sc.a[r] * sc.h / p.mu : 0.0;
    }
}

__device__ __forceinline__ void split_hi_lo(double v, float &hi, float &lo)
{
    hi = (float)v;
    lo = (float)(v - (double)hi);
}

__device__ __forceinline__ double frac1(double v) { return v - rint(v); }

constexpr double kPi = 3.14159265358979323846;
constexpr double kInv4Pi = 0.079577471545947667884;  // 1/(4 pi)
constexpr double kInv2Pi = 0.15915494309189533577;   // 1/(2 pi)

// the phase record of 1D sub-stage j (turns per integer index, see above)
// per-instance factors of the turn coefficients: dx^2/(4 pi), xc dx/(2 pi),
// xc^2/(4 pi), pi/L^2, h/(2 pi)
struct RecScale {
    double k2, k1, k0, g, sb;
};
__device__ __forceinline__ RecScale rec_scale(const DevInst &p, const SchedConst &sc)
{
    RecScale c;
    c.k2 = p.dx[0] * p.dx[0] * kInv4Pi;
    c.k1 = p.xc[0] * p.dx[0] * kInv2Pi;
    c.k0 = p.xc[0] * p.xc[0] * kInv4Pi;
    c.g = kPi / (p.len[0] * p.len[0]);
    c.sb = sc.h * kInv2Pi;
    return c;
}

template <typename RecT, int SPLIT>
__device__ __forceinline__ void record1d(const DevInst &p, const SchedConst &sc, const RecScale &c, double t0, int j,
                                         int nstage, const StageFGE *__restrict__ fge_i, RecT *out, unsigned *status)
{
    double kappa, bs, g;
    merged_coeffs<SPLIT>(p, 1, 0, sc, t0, j, nstage, fge_i, kappa, bs, g);
    const double K2 = kappa * c.k2;
    const double G = g * c.g;
    const double SB = bs * c.sb;
    // the terms of an off-centre box (half of a record's FP64 work)
    double K1 = 0.0, K0 = 0.0;
    if (c.k1 != 0.0) {
        K1 = kappa * c.k1;
        K0 = frac1(kappa * c.k0);
    }
    if (!isfinite(K2) || !isfinite(G) || !isfinite(K1)) atomicOr(status, (unsigned)ST_NONFINITE);
    RecT r;
    if constexpr (sizeof(RecT) == sizeof(RecF)) {
        split_hi_lo(K2, r.k2hi, r.k2lo);
        r.k1hi = r.k1lo = r.k0 = 0.0f;
        if (c.k1 != 0.0) {
            split_hi_lo(K1, r.k1hi, r.k1lo);
            r.k0 = (float)K0;
        }
        r.sb2pi = (float)SB;
        split_hi_lo(G, r.ghi, r.glo);
    } else {
        r.k2 = K2;
        r.k1 = K1;
        r.k0 = K0;
        r.sb2pi = SB;
        r.g = G;
        r.pad = 0.0;
    }
    *out = r;
}

}  // namespace hfs
