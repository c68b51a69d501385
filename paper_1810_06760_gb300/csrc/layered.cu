// A7: beams in a medium of homogeneous layers (Sec. 3.1) between parallel planes, concentric spheres or
// undulating surfaces.  Inside a layer grad c = 0, so a beam moves on a straight line; a step that crosses an
// interface is split at the crossing, where the beam is replaced by its reflected and transmitted P and
// S children (Snell's law, plane-wave continuity of displacement and traction, and the dzQ/dzP jump of
// Eq. Inter_DzQDzP; at a sphere all of it in the local tangent-normal frame of the crossing point), and
// every child finishes the step.  Children are appended to the beam arrays with an atomic counter; the
// parent's slot goes to its first child.
#include <algorithm>
#include <cmath>

#include "fga_beam.cuh"
#include "gather.cuh"
#include "straight.cuh"

namespace fga {

namespace {

struct Cd {
    double r, i;
};
__device__ __forceinline__ Cd cadd(Cd a, Cd b) { return {a.r + b.r, a.i + b.i}; }
__device__ __forceinline__ Cd csub2(Cd a, Cd b) { return {a.r - b.r, a.i - b.i}; }
__device__ __forceinline__ Cd cmulx(Cd a, Cd b) { return {a.r * b.r - a.i * b.i, a.r * b.i + a.i * b.r}; }
__device__ __forceinline__ Cd cscale(Cd a, double s) { return {a.r * s, a.i * s}; }
__device__ __forceinline__ double cabs2(Cd a) { return a.r * a.r + a.i * a.i; }

// Layer speed of a beam (bits 4-7 of its flags hold its layer).
template <typename R> __device__ __forceinline__ R layer_speed(const ModelDev &M, int wave, int lay) {
    return wave ? mp<R>(M.lcs[lay], M.flcs[lay]) : mp<R>(M.lcp[lay], M.flcp[lay]);
}

// Children of an event (w = 0 reflected P, 1 reflected S, 2 transmitted P, 3 transmitted S), FP64.
struct EventOut {
    int n;
    int slot[4], flags[4];
    double P[4][3];
    Cd a0[4], a1[4];        // P: a0; S: (a_sv, a_sh) in the child's own frame
    double gh[4], f22[4];   // the jump of dzQ, dzP: g = gh Ph + (f22 - 1) n
    double Ph[3];           // the part of P along the interface
};

// cos and sin of the angle, seen along P, from the S frame of P (reference e1 or e3) to the unit vector nsh normal to P:
// nsh = sin N_sv + cos N_sh
__device__ __forceinline__ void frame_angle(const double P[3], double pn, bool r1, const double nsh[3], double &c, double &s) {
    double v[3];
    if (r1) {
        v[0] = 0.0;
        v[1] = -P[2];
        v[2] = P[1];
    } else {
        v[0] = -P[1];
        v[1] = P[0];
        v[2] = 0.0;
    }
    const double iv = rsqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    c = iv * (v[0] * nsh[0] + v[1] * nsh[1] + v[2] * nsh[2]);
    s = iv / pn *
        ((v[1] * P[2] - v[2] * P[1]) * nsh[0] + (v[2] * P[0] - v[0] * P[2]) * nsh[1] + (v[0] * P[1] - v[1] * P[0]) * nsh[2]);
}

// The scattering at an interface with unit normal n (e3 for SHAPE 0) between layer la (incident side) and lb; y holds
// the incident state.  Polarisations: P along P/|P|; SH along nsh = n x P/|n x P| (common to all waves of the event; e2
// at normal incidence); SV along nsh x P/|P|.  Displacement and traction on the interface are continuous.
//
// In the plane of P and n the six conditions separate.  With p = |P_h|, normal components zeta (P) and eta (S) of every
// medium, and S amplitudes signed by the wave's direction along n, the pairs (u_h, sigma_nn) and (u_n, sigma_hn) of
// waves to either side differ only in sign, so that, amplitudes divided by |P| of their wave,
//   M_a (i + r) = M_b t,  N_a (i - r) = N_b t,  M = [p 1; G -2 mu p] diag(1, eta),  N = [1 -p; 2 mu p G] diag(zeta, 1),
//   G = rho om^2 - 2 mu p^2,  det = -+ rho om^2,
// a 2x2 complex system for the transmitted P and SV; SH is a ratio.  About 200 FP64 operations in a short chain where
// elimination on the 6x6 complex system takes 3,000 in local memory (an event kernel runs few warps, and the FP64 pipe
// issues one warp instruction in 16 cycles: the chain is what bounds it).
template <typename R, int SHAPE>
__device__ __forceinline__ bool interface_event(const ModelDev &M, int fl, const R *y, const double n[3], int lb,
                                                double rel_min, EventOut &ev) {
    const int la = (fl >> 4) & 15, cls = fl & FL_CLASS_MASK, wave = cls >= 2;
    const double sgn = (cls & 1) ? -1.0 : 1.0;
    const double P[3] = {(double)y[F_P], (double)y[F_P + 1], (double)y[F_P + 2]};
    const double cin = wave ? M.lcs[la] : M.lcp[la];
    const double pin = sqrt(P[0] * P[0] + P[1] * P[1] + P[2] * P[2]), om = cin * pin;
    const double pz = SHAPE == 0 ? P[2] : P[0] * n[0] + P[1] * n[1] + P[2] * n[2];
#pragma unroll
    for (int d = 0; d < 3; d++) ev.Ph[d] = SHAPE == 0 ? (d < 2 ? P[d] : 0.0) : P[d] - pz * n[d];
    const double ph2 = ev.Ph[0] * ev.Ph[0] + ev.Ph[1] * ev.Ph[1] + ev.Ph[2] * ev.Ph[2];
    const double ph = sqrt(ph2);
    double nsh[3] = {0.0, 1.0, 0.0};
    if (SHAPE == 0) {
        if (ph2 > 0.0) {
            const double ip = rsqrt(ph2);
            nsh[0] = -ip * P[1];
            nsh[1] = ip * P[0];
        }
    } else {
        // Near normal incidence n x P is rounding, part of it along n.  That part is taken out and what is left is
        // normalised by itself, so that nsh is a unit vector normal to n and P, whose direction in the interface does not
        // matter there (divided by |P_h|, rounding along n and all, S beams lost up to all of their amplitude); where
        // nothing but rounding is left, any direction in the interface.
        double v[3] = {n[1] * P[2] - n[2] * P[1], n[2] * P[0] - n[0] * P[2], n[0] * P[1] - n[1] * P[0]};
        const double vn = v[0] * n[0] + v[1] * n[1] + v[2] * n[2];
#pragma unroll
        for (int d = 0; d < 3; d++) v[d] -= vn * n[d];
        const double v2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
        if (v2 > 1e-28 * pin * pin) {
            const double iv = rsqrt(v2);
#pragma unroll
            for (int d = 0; d < 3; d++) nsh[d] = iv * v[d];
        } else {
            double Rl[9];
            frame_from_normal(n, Rl);
            for (int d = 0; d < 3; d++) nsh[d] = Rl[3 + d];
        }
    }
    // incident amplitudes along P/|P|, or along SV and SH of the interface
    const Cd a0 = {(double)y[F_A0], (double)y[F_A0 + 1]}, a1 = {(double)y[F_A1], (double)y[F_A1 + 1]};
    double ain2 = cabs2(a0);
    Cd iP = a0, iS = {0.0, 0.0}, iH = {0.0, 0.0};
    if (wave) {
        iP = {0.0, 0.0};
        iS = a0;
        iH = a1;
        ain2 += cabs2(a1);
        if (SHAPE != 0 || (fl & FL_REF_E1) || !(ph2 > 0.0)) {
            double c, s;
            frame_angle(P, pin, (fl & FL_REF_E1) != 0, nsh, c, s);
            iS = csub2(cscale(a0, c), cscale(a1, s));
            iH = cadd(cscale(a0, s), cscale(a1, c));
        }
    }
    const double sz = pz >= 0.0 ? 1.0 : -1.0;
    double kw[4], cw[4], zr[4];   // |P|, speed and |normal component| of the waves
    bool prop[4];
    Cd z[4];
#pragma unroll
    for (int w = 0; w < 4; w++) {
        const int L = w >= 2 ? lb : la;
        cw[w] = w & 1 ? M.lcs[L] : M.lcp[L];
        kw[w] = om / cw[w];
        const double pz2 = kw[w] * kw[w] - ph2;
        prop[w] = pz2 >= 0.0;
        zr[w] = sqrt(fabs(pz2));
        z[w] = prop[w] ? Cd{zr[w], 0.0} : Cd{0.0, sgn * zr[w]};   // decays away from the interface
    }
    const double mua = M.lrho[la] * M.lcs[la] * M.lcs[la], mub = M.lrho[lb] * M.lcs[lb] * M.lcs[lb];
    const double om2 = om * om, Ga = M.lrho[la] * om2 - 2.0 * mua * ph2, Gb = M.lrho[lb] * om2 - 2.0 * mub * ph2;
    const double iD = 1.0 / (M.lrho[la] * om2);
    const double u = (2.0 * mua * ph2 + Gb) * iD, v = (Ga + 2.0 * mub * ph2) * iD, x = 2.0 * ph * (mua - mub) * iD,
                 wq = ph * (Ga - Gb) * iD;
    const Cd jP = cscale(iP, 1.0 / kw[0]), jS = cscale(iS, sz / kw[1]);
    const Cd A11 = cadd(cscale(z[0], u), cscale(z[2], v)), A22 = cadd(cscale(z[3], v), cscale(z[1], u));
    Cd A12 = cscale(cmulx(z[0], z[3]), x), A21 = cscale(cmulx(z[1], z[2]), -x);
    A12.r -= wq;
    A21.r += wq;
    const Cd det = csub2(cmulx(A11, A22), cmulx(A12, A21));
    const Cd denH = cadd(cscale(z[1], mua), cscale(z[3], mub));
    const double d2 = cabs2(det), h2 = cabs2(denH);
    if (!(d2 > 0.0) || !(h2 > 0.0)) return false;
    const Cd id = {det.r / d2, -det.i / d2};
    const Cd b1 = cscale(cmulx(z[0], jP), 2.0), b2 = cscale(cmulx(z[1], jS), 2.0);
    const Cd tP = cmulx(csub2(cmulx(b1, A22), cmulx(A12, b2)), id), tS = cmulx(csub2(cmulx(A11, b2), cmulx(A21, b1)), id);
    const Cd rP = csub2(cadd(cscale(tP, u), cscale(cmulx(z[3], tS), x)), jP);
    const Cd rS = csub2(cadd(jS, cscale(cmulx(z[2], tP), x)), cscale(tS, u));
    Cd tH = {0.0, 0.0}, rH = {0.0, 0.0};
    if (wave) {
        const Cd ih = {denH.r / h2, -denH.i / h2};
        tH = cmulx(cmulx(cscale(z[1], 2.0 * mua), iH), ih);
        rH = csub2(tH, iH);
    }
    const Cd am[4] = {cscale(rP, kw[0]), cscale(rS, -sz * kw[1]), cscale(tP, kw[2]), cscale(tS, sz * kw[3])};
    const int gen = (fl >> 8) & 15;
    const double ipz = 1.0 / pz, icin2 = 1.0 / (cin * cin);
    int m = 0;
#pragma unroll
    for (int w = 0; w < 4; w++) {
        const int sw = w & 1, trans = w >= 2;
        Cd b0 = am[w], b1c = sw ? (trans ? tH : rH) : Cd{0.0, 0.0};
        const double amag2 = cabs2(b0) + cabs2(b1c);
        if (!prop[w] || !(amag2 >= rel_min * rel_min * ain2) || amag2 == 0.0) continue;
        const double zz = trans ? sz * zr[w] : -sz * zr[w];
        double Pc[3];
#pragma unroll
        for (int d = 0; d < 3; d++) Pc[d] = SHAPE == 0 ? (d < 2 ? P[d] : zz) : ev.Ph[d] + zz * n[d];
        int flc = (sw ? 2 : 0) | (cls & 1) | ((trans ? lb : la) << 4) | ((gen + 1) << 8) | (fl & (3 << FL_ROOT_SHIFT));
        if (sw) {
            // SV/SH of the interface -> the child's own frame (e3 unless its P is near vertical)
            const double h = Pc[0] * Pc[0] + Pc[1] * Pc[1];
            const bool r1 = h < 0.01 * (h + Pc[2] * Pc[2]);
            if (r1) flc |= FL_REF_E1;
            if (SHAPE != 0 || r1) {
                double c, s;
                frame_angle(Pc, kw[w], r1, nsh, c, s);
                const Cd t0 = b0, t1 = b1c;
                b0 = cadd(cscale(t0, c), cscale(t1, s));
                b1c = csub2(cscale(t1, c), cscale(t0, s));
            }
        }
        ev.slot[m] = w;
        ev.flags[m] = flc;
        ev.a0[m] = b0;
        ev.a1[m] = b1c;
        const double kappa = cw[w] * cw[w] * icin2;
        ev.gh[m] = (kappa - 1.0) * ipz;
        ev.f22[m] = kappa * zz * ipz;
#pragma unroll
        for (int d = 0; d < 3; d++) ev.P[m][d] = Pc[d];
        m++;
    }
    ev.n = m;
    return true;
}

// Child k of the event into out[] (NF reals): Q at the crossing, new P, dzQ F, dzP F^{-T}, amplitudes.  F is I but
// for its row along the normal, so in any frame dzQ' = dzQ + (dzQ n) g^T and dzP' = dzP - (dzP g) n^T / f22.
template <typename R, int SHAPE>
__device__ __forceinline__ void make_child(const R *yc, const EventOut &ev, const double n[3], int k, R *out) {
#pragma unroll
    for (int d = 0; d < 3; d++) out[F_Q + d] = yc[F_Q + d];
    const double gh = ev.gh[k], f22 = ev.f22[k], if22 = 1.0 / f22;
    const double g0 = gh * ev.Ph[0] + (SHAPE == 0 ? 0.0 : (f22 - 1.0) * n[0]),
                 g1 = gh * ev.Ph[1] + (SHAPE == 0 ? 0.0 : (f22 - 1.0) * n[1]),
                 g2 = SHAPE == 0 ? 0.0 : gh * ev.Ph[2] + (f22 - 1.0) * n[2];
#pragma unroll
    for (int m = 0; m < 3; m++) {
#pragma unroll
        for (int c = 0; c < 2; c++) {  // re, im
            const int e0 = 2 * (3 * m) + c, e1 = e0 + 2, e2 = e0 + 4;
            const double q0 = yc[F_DQ + e0], q1 = yc[F_DQ + e1], q2 = yc[F_DQ + e2];
            const double p0 = yc[F_DP + e0], p1 = yc[F_DP + e1], p2 = yc[F_DP + e2];
            if (SHAPE == 0) {
                out[F_DQ + e0] = (R)(q0 + q2 * g0);
                out[F_DQ + e1] = (R)(q1 + q2 * g1);
                out[F_DQ + e2] = (R)(q2 * f22);
                out[F_DP + e0] = yc[F_DP + e0];
                out[F_DP + e1] = yc[F_DP + e1];
                out[F_DP + e2] = (R)((p2 - p0 * g0 - p1 * g1) * if22);
            } else {
                const double qn = q0 * n[0] + q1 * n[1] + q2 * n[2], pg = -if22 * (p0 * g0 + p1 * g1 + p2 * g2);
                out[F_DQ + e0] = (R)(q0 + qn * g0);
                out[F_DQ + e1] = (R)(q1 + qn * g1);
                out[F_DQ + e2] = (R)(q2 + qn * g2);
                out[F_DP + e0] = (R)(p0 + pg * n[0]);
                out[F_DP + e1] = (R)(p1 + pg * n[1]);
                out[F_DP + e2] = (R)(p2 + pg * n[2]);
            }
        }
    }
#pragma unroll
    for (int d = 0; d < 3; d++) out[F_P + d] = (R)ev.P[k][d];
    out[F_A0] = (R)ev.a0[k].r;
    out[F_A0 + 1] = (R)ev.a0[k].i;
    out[F_A1] = (R)ev.a1[k].r;
    out[F_A1 + 1] = (R)ev.a1[k].i;
}

// Spherical layers (interfaces |x - c| = rho_i, rho_i = -zif[i] decreasing): the first crossing of the
// straight path q0 -> q1 of one step (a beam moves on a line in a homogeneous layer) with a sphere that
// bounds layer L, s(th) = q0 - c + th d, d = q1 - q0, |s(th)|^2 = a th^2 + b th + |q0 - c|^2.  The inner
// sphere is met when the path heads inward (b < 0) and the smaller root, 2 c0 / (-b + sqrt D), lies below
// 1 (a path may dip into it and leave again within one step); the outer sphere bounds a convex ball, so
// only an end point beyond it means a crossing, at the positive root.  Returns false without a crossing,
// else the fraction th of the step, the layer lb entered and the radius crossed.
__device__ __noinline__ bool shell_crossing(const ModelDev &M, int L, const double q0[3], const double q1[3], double &th, int &lb,
                               double &rho) {
    double s0[3], d[3], s1[3];
    for (int c = 0; c < 3; c++) {
        s0[c] = q0[c] - M.ctr[c];
        s1[c] = q1[c] - M.ctr[c];
        d[c] = q1[c] - q0[c];
    }
    const double a = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    const double b = 2.0 * (s0[0] * d[0] + s0[1] * d[1] + s0[2] * d[2]);
    const double ss = s0[0] * s0[0] + s0[1] * s0[1] + s0[2] * s0[2];
    bool hit = false;
    if (L < M.nlay - 1) {
        const double r = -M.zif[L];
        const double c0 = ss - r * r, D = b * b - 4.0 * a * c0;
        if (b < 0.0 && D >= 0.0) {
            const double t = 2.0 * c0 / (-b + sqrt(D));
            if (t < 1.0) {
                th = t;
                lb = L + 1;
                rho = r;
                hit = true;
            }
        }
    }
    if (L > 0) {
        const double r = -M.zif[L - 1];
        if (s1[0] * s1[0] + s1[1] * s1[1] + s1[2] * s1[2] > r * r) {
            const double c0 = ss - r * r, D = fmax(b * b - 4.0 * a * c0, 0.0);
            const double t = b <= 0.0 ? (-b + sqrt(D)) / (2.0 * a) : -2.0 * c0 / (b + sqrt(D));
            if (!hit || t < th) {
                th = t;
                lb = L - 1;
                rho = r;
                hit = true;
            }
        }
    }
    return hit;
}

// FP32 screen for spherical layers: true when the straight path q0 -> q1 certainly meets no sphere of
// layer L, i.e. the end point lies inside the enclosing sphere and the path's closest approach to the
// centre lies outside the inner one, each with a relative margin of 1e-5 on r^2.
__device__ __forceinline__ bool shell_clear(const ModelDev &M, int L, const float *q0, const float *q1) {
    const float c0 = (float)M.ctr[0], c1 = (float)M.ctr[1], c2 = (float)M.ctr[2];
    const float s0[3] = {q0[0] - c0, q0[1] - c1, q0[2] - c2};
    const float d[3] = {q1[0] - q0[0], q1[1] - q0[1], q1[2] - q0[2]};
    const float r0 = s0[0] * s0[0] + s0[1] * s0[1] + s0[2] * s0[2];
    const float a = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    const float b = 2.0f * (s0[0] * d[0] + s0[1] * d[1] + s0[2] * d[2]);
    if (L > 0) {
        const float ro = M.fzif[L - 1];                      // minus the enclosing radius
        const float r1 = r0 + b + a;                         // |q1 - c|^2
        if (!(r1 < ro * ro * (1.0f - 1e-5f))) return false;
    }
    if (L < M.nlay - 1) {
        const float ri = M.fzif[L];
        float t = b < 0.0f ? -b / (2.0f * a) : 0.0f;         // closest approach on the path
        t = t > 1.0f ? 1.0f : t;
        const float rmin = r0 + t * (b + a * t);
        if (!(rmin > ri * ri * (1.0f + 1e-5f))) return false;
    }
    return true;
}
__device__ __forceinline__ bool shell_clear(const ModelDev &, int, const double *, const double *) { return false; }

// Undulating layers: height of interface i above (x1, x2), and its slopes dh/dx1, dh/dx2.
__device__ __forceinline__ double surf_cos(const ModelDev &M, const double *q) { return cos(M.uk[0] * q[0]) * cos(M.uk[1] * q[1]); }
__device__ __forceinline__ double surf_at(const ModelDev &M, int i, double x1, double x2, double &h1, double &h2) {
    double s1, c1, s2, c2;
    sincos(M.uk[0] * x1, &s1, &c1);
    sincos(M.uk[1] * x2, &s2, &c2);
    h1 = -M.uamp[i] * M.uk[0] * s1 * c2;
    h2 = -M.uamp[i] * M.uk[1] * c1 * s2;
    return M.zif[i] + M.uamp[i] * (c1 * c2);
}

// FP32 screen for undulating layers: true when the end point q1 lies clearly between the interfaces that
// bound layer L (by a margin far above the FP32 rounding of the heights, which grows with the phase
// k |x| of the cosines).
__device__ __forceinline__ bool surf_clear(const ModelDev &M, int L, const float *q1) {
    const float ph = M.fuk[0] * fabsf(q1[0]) + M.fuk[1] * fabsf(q1[1]);
    float mid[2], amp[2], mar[2];   // lower and upper interface of the layer: mean depth, amplitude, margin
#pragma unroll
    for (int e = 0; e < 2; e++) {
        const int i = e == 0 ? L : L - 1;
        const bool there = i >= 0 && i < M.nlay - 1;
        mid[e] = there ? M.fzif[i] : (e == 0 ? INFINITY : -INFINITY);
        amp[e] = there ? M.fuamp[i] : 0.0f;
        mar[e] = there ? 1e-4f * (1.0f + fabsf(mid[e]) + fabsf(amp[e])) + 2e-6f * fabsf(amp[e]) * ph : 0.0f;
    }
    // outside both interfaces' bands of depth no height is needed
    if (q1[2] < mid[0] - fabsf(amp[0]) - mar[0] && q1[2] >= mid[1] + fabsf(amp[1]) + mar[1]) return true;
    const float cc = cosf(M.fuk[0] * q1[0]) * cosf(M.fuk[1] * q1[1]);
    return q1[2] < mid[0] + amp[0] * cc - mar[0] && q1[2] >= mid[1] + amp[1] * cc + mar[1];
}
__device__ __forceinline__ bool surf_clear(const ModelDev &, int, const double *) { return false; }

// The step's end point q1 on or below the lower interface of layer L, or above the upper one: a crossing.
__device__ __forceinline__ bool surf_met(const ModelDev &M, int L, bool down, const double q1[3], double cc1, double &g1) {
    const int i = down ? L : L - 1;
    if (i < 0 || i > M.nlay - 2) return false;
    g1 = q1[2] - (M.zif[i] + M.uamp[i] * cc1);
    return down ? g1 >= 0.0 : g1 < 0.0;
}
__device__ __noinline__ bool surf_crosses(const ModelDev &M, int L, const double q1[3]) {
    const double cc1 = surf_cos(M, q1);
    double g;
    return surf_met(M, L, true, q1, cc1, g) || surf_met(M, L, false, q1, cc1, g);
}

// Undulating layers: the first crossing of the straight path q0 -> q1 of one step with an interface that
// bounds layer L.  An end point on or below the lower interface (above the upper one) means a crossing;
// g(th) = x3(th) - h(x1(th), x2(th)) then changes sign on [0, 1] and its root is found by Newton's method
// kept inside a shrinking bracket (bisection where a Newton step leaves it; at most 100 iterations).  A
// start already beyond the interface (no sign change) takes the root of g's linear interpolation (the start
// itself when g does not change along the path).
// Returns false without a crossing, else th, the layer lb entered and the interface index.
__device__ __noinline__ bool surf_crossing(const ModelDev &M, int L, const double q0[3], const double q1[3], double &th, int &lb,
                              int &iface) {
    const double d[3] = {q1[0] - q0[0], q1[1] - q0[1], q1[2] - q0[2]};
    const double cc0 = surf_cos(M, q0), cc1 = surf_cos(M, q1);
    bool hit = false;
    for (int side = 0; side < 2; side++) {
        const bool down = side == 0;
        double g1;
        if (!surf_met(M, L, down, q1, cc1, g1)) continue;
        const int i = down ? L : L - 1;
        const double g0 = q0[2] - (M.zif[i] + M.uamp[i] * cc0);
        double t;
        if ((g0 < 0.0) == down) {
            double lo = 0.0, hi = 1.0, glo = g0;   // g(lo) and g(hi) of opposite signs
            t = g0 / (g0 - g1);
            for (int it = 0; it < 100 && hi - lo > 1e-15; it++) {
                double h1, h2;
                const double g = q0[2] + t * d[2] - surf_at(M, i, q0[0] + t * d[0], q0[1] + t * d[1], h1, h2);
                if (g == 0.0) break;
                if ((g < 0.0) == (glo < 0.0)) {
                    lo = t;
                    glo = g;
                } else {
                    hi = t;
                }
                const double dg = d[2] - h1 * d[0] - h2 * d[1];
                double tn = dg != 0.0 ? t - g / dg : 0.5 * (lo + hi);
                if (!(tn > lo && tn < hi)) tn = 0.5 * (lo + hi);
                const double step = fabs(tn - t);
                t = tn;
                if (step < 1e-12) break;   // the next correction is of the order of its square
            }
        } else {
            t = g0 != g1 ? g0 / (g0 - g1) : 0.0;   // no motion across the surface: the start itself
        }
        if (!hit || t < th) {
            th = t;
            lb = down ? L + 1 : L - 1;
            iface = i;
            hit = true;
        }
    }
    return hit;
}

}  // namespace

// Write child ce (with its Q compensation) of the beam in slot b: the first child takes the parent's slot,
// the others are appended (atomic counter); children beyond cap are counted in counts[1].  Returns the slot
// (-1 for a child beyond cap).
template <typename R>
__device__ int64_t store_child(R *__restrict__ st, int32_t *__restrict__ flags, int32_t *__restrict__ ids,
                               long long *__restrict__ path, int64_t cap, unsigned long long *__restrict__ counts,
                               int64_t b, int k, const R *ce, const R *qch, int flc, int32_t id, long long pp, int slot) {
    int64_t dst = b;
    if (k > 0) {
        dst = (int64_t)atomicAdd(&counts[0], 1ull);
        if (dst >= cap) {
            atomicAdd(&counts[1], 1ull);
            return -1;
        }
    }
#pragma unroll
    for (int f = 0; f < NF; f++) st[(int64_t)f * cap + dst] = ce[f];
#pragma unroll
    for (int d = 0; d < 3; d++) st[(int64_t)(F_QC + d) * cap + dst] = qch[d];
    flags[dst] = flc;
    ids[dst] = id;
    path[dst] = pp * 4 + slot + 1;
    return dst;
}

// Interfaces that bound layer L of a planar medium.
template <typename R> struct Planes {
    R top, bot;
    __device__ __forceinline__ Planes(const ModelDev &M, int L)
        : top(L > 0 ? mp<R>(M.zif[L - 1], M.fzif[L - 1]) : -R(INFINITY)),
          bot(L < M.nlay - 1 ? mp<R>(M.zif[L], M.fzif[L]) : R(INFINITY)) {}
};

// Does the step q0 -> q1 (compensations c0, c1) meet an interface of layer L?  Planes: the end point.  Curved
// layers: FP32 steps that stay clear of the interfaces by a margin far above the rounding of the screen are
// decided by the screen, the rest by the exact FP64 test, which with WHERE also gives the crossing.
struct Crossing {
    double th, rho;
    int lb, iface;
};
template <typename R, int SHAPE, bool WHERE>
__device__ __forceinline__ bool step_crosses(const ModelDev &M, int L, const Planes<R> &pl, const R *q0, const R *c0,
                                             const R *q1, const R *c1, Crossing &x) {
    if (SHAPE == 0) return q1[2] < pl.top || q1[2] >= pl.bot;
    if (sizeof(R) == 4 && (SHAPE == 1 ? shell_clear(M, L, q0, q1) : surf_clear(M, L, q1))) return false;
    double a[3], b[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        a[d] = (double)q0[d] - (double)c0[d];
        b[d] = (double)q1[d] - (double)c1[d];
    }
    if (SHAPE == 1) return shell_crossing(M, L, a, b, x.th, x.lb, x.rho);
    return WHERE ? surf_crossing(M, L, a, b, x.th, x.lb, x.iface) : surf_crosses(M, L, b);
}

// At most m steps of a beam from its expansion S, the first at time t0 of it: Q, its compensation and the amplitudes
// in y, qc (dzQ is left to the caller).  Returns the steps made; open: no interface was met.
template <typename R, int SHAPE>
__device__ __forceinline__ int straight_run(const ModelDev &M, int L, const Planes<R> &pl, const Straight<R> &S, R t0, R *y,
                                            R *qc, R dt, int m, bool force_first, bool &open) {
    C2<R> g1 = straight_gamma<R>(S, t0);
    int i = 0;
    for (; i < m; i++) {
        R q[3] = {y[F_Q], y[F_Q + 1], y[F_Q + 2]}, qn[3] = {qc[0], qc[1], qc[2]};
        straight_q<R>(S, dt, q, qn);
        Crossing x;
        if (!force_first && step_crosses<R, SHAPE, false>(M, L, pl, y + F_Q, qc, q, qn, x)) {
            open = false;
            break;
        }
        force_first = false;
        const R t = t0 + R(i) * dt;
        const C2<R> g2 = straight_gamma<R>(S, t + R(0.5) * dt), g4 = straight_gamma<R>(S, t + dt);
        straight_amplitudes<R>(y, straight_gain<R>(dt, g1, g2, g4));
        g1 = g4;
#pragma unroll
        for (int d = 0; d < 3; d++) {
            y[F_Q + d] = q[d];
            qc[d] = qn[d];
        }
    }
    return i;
}

// Steps s .. nsteps-1 of a beam up to the first one that meets an interface; returns that step's index (nsteps
// without one), the state at its start in y, qc.  Every step but that one is the closed form of straight.cuh.
// lead > 0: a part of a step of that length comes first (a child's way from its interface to the step's end).
template <typename R, int SHAPE>
__device__ __forceinline__ int layered_run(const ModelDev &M, int fl, R *y, R *qc, R dt, int s, int nsteps,
                                           bool force_first, bool part = false, R lead = R(0)) {
    const int wave = (fl & FL_CLASS_MASK) >= 2, L = (fl >> 4) & 15;
    const R sg = (fl & 1) ? R(-1) : R(1), c = layer_speed<R>(M, wave, L);
    const Planes<R> pl(M, L);
    bool open = true;
    while (open && (part || s < nsteps)) {
        R B[18];
        Straight<R> S;
        straight_setup<R>(sg, c, y, B, S);
        R t0 = R(0);
        if (part) {
            straight_part<R>(S, lead, y, qc);
            t0 = lead;
            part = false;
        }
        const int i = straight_run<R, SHAPE>(M, L, pl, S, t0, y, qc, dt, min(STRAIGHT_RENEW, nsteps - s), force_first, open);
        force_first = false;
        const R T = t0 + R(i) * dt;
#pragma unroll
        for (int f = 0; f < 18; f++) y[F_DQ + f] += T * B[f];
        s += i;
    }
    return s;
}

template <typename R>
__device__ __forceinline__ void load_beam(const R *__restrict__ st, int64_t cap, int64_t b, R *y, R *qc) {
#pragma unroll
    for (int f = 0; f < NF; f++) y[f] = st[(int64_t)f * cap + b];
#pragma unroll
    for (int d = 0; d < 3; d++) qc[d] = st[(int64_t)(F_QC + d) * cap + b];
}

// append (beam slot, step) to an event list: one atomic per converged group of lanes
__device__ __forceinline__ void push_event(int2 *__restrict__ list, unsigned *__restrict__ n, int64_t b, int s) {
    const unsigned mask = __activemask(), lane = threadIdx.x & 31;
    const int lead = __ffs(mask) - 1;
    unsigned at = 0;
    if ((int)lane == lead) at = atomicAdd(n, (unsigned)__popc(mask));
    at = __shfl_sync(mask, at, lead) + __popc(mask & ((1u << lane) - 1u));
    list[at] = make_int2((int)b, s);
}

// A group of nsteps steps, first part: every live beam advances until the group's end or until a step that
// meets an interface; such beams are listed with their step (or die, past their last allowed interface).
// One state stream per group instead of one per step: 49 reals read and 28 written per beam (P and dzP stay),
// which bounds it.  442 k beams growing to 0.9 M, 300 steps in groups of 5, FP32: 69.6 ms (a launch per step
// with four right-hand sides, events inside) -> 3.2 ms of these kernels and 3.8 ms of event kernels; with
// undulating interfaces (an FP64 test of the end point where the FP32 screen cannot decide) 187 -> 5.2 and 7.9 ms.
// The grid strides over the live beams: blocks for the whole reserved capacity, eight times the first population, cost 0.6 ms.
template <typename R, int SHAPE>
__global__ void __launch_bounds__(128) layered_run_kernel(ModelDev M, R *__restrict__ st, int32_t *__restrict__ flags,
                                                         int64_t cap, const unsigned long long *__restrict__ counts,
                                                         int64_t first, int64_t end, R dt, int nsteps, int gmax,
                                                         int2 *__restrict__ list, unsigned *__restrict__ nlist) {
    const int64_t n = min((unsigned long long)end, counts[0]);   // slots first .. end - 1
    for (int64_t b = first + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < n; b += (int64_t)gridDim.x * blockDim.x) {
        const int fl = flags[b];
        if (fl & FL_DEAD) continue;
        R y[NF], qc[3];
        load_beam<R>(st, cap, b, y, qc);
        const int s = layered_run<R, SHAPE>(M, fl, y, qc, dt, 0, nsteps, false);
#pragma unroll
        for (int f = 0; f < 3; f++) st[(int64_t)f * cap + b] = y[f];
#pragma unroll
        for (int f = F_DQ; f < F_DP; f++) st[(int64_t)f * cap + b] = y[f];
#pragma unroll
        for (int f = F_A0; f < NF; f++) st[(int64_t)f * cap + b] = y[f];
#pragma unroll
        for (int d = 0; d < 3; d++) st[(int64_t)(F_QC + d) * cap + b] = qc[d];
        if (s == nsteps) continue;
        if (((fl >> 8) & 15) >= gmax)
            flags[b] = fl | FL_DEAD;
        else
            push_event(list, nlist, b, s);
    }
}

// The listed beams: the event of step s at its interface, then every child finishes that step and advances
// like the beams of layered_run_kernel; children that meet another interface go to the next list.  A thread
// per event, in a kernel of its own so that whole warps are on events (inside the step kernel one lane of a warp held
// the other 31).  A few thousand events a launch are one or two warps per SM: the length of an event's FP64 chain
// bounds it.  With the 6x6 system of an event eliminated in general and the state rotated to the interface's frame and
// back for every child these kernels took 8.7 ms (flat) and 22.1 ms (undulating) where they now take 3.8 and 7.9.
//
// In curved layers (SHAPE 1: spheres, SHAPE 2: undulating interfaces) the crossing is put on the interface in
// FP64 (radially onto the sphere, vertically onto the undulating surface; its FP32 rounding goes to the Q
// compensation) and the event runs with the interface's normal there (Sec. 3.1: the tangent plane stands in for the
// interface), in global coordinates.
template <typename R, int SHAPE>
__global__ void __launch_bounds__(64) layered_event_kernel(ModelDev M, R *__restrict__ st, int32_t *__restrict__ flags,
                                                          int32_t *__restrict__ ids, long long *__restrict__ path,
                                                          int64_t cap, unsigned long long *__restrict__ counts, R dt,
                                                          int nsteps, int gmax, double rel_min,
                                                          const int2 *__restrict__ list, const unsigned *__restrict__ nlist,
                                                          int2 *__restrict__ next, unsigned *__restrict__ nnext) {
    const unsigned n = *nlist;
    for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        const int64_t b = list[e].x;
        int s = list[e].y;
        const int fl = flags[b];
        const int L = (fl >> 4) & 15;
        const R sg = (fl & 1) ? R(-1) : R(1), c = layer_speed<R>(M, (fl & FL_CLASS_MASK) >= 2, L);
        const Planes<R> pl(M, L);
        R y[NF], qc[3];
        load_beam<R>(st, cap, b, y, qc);
        Crossing x{0.0, 0.0, L, 0};
        bool hit = false;
        R B[18];
        Straight<R> S;
        while (s < nsteps) {
            // the step's end point as layered_run forms it
            R q[3] = {y[F_Q], y[F_Q + 1], y[F_Q + 2]}, qn[3] = {qc[0], qc[1], qc[2]};
            straight_setup<R>(sg, c, y, B, S);
            straight_q<R>(S, dt, q, qn);
            hit = step_crosses<R, SHAPE, true>(M, L, pl, y + F_Q, qc, q, qn, x);
            if (hit) {
                if (SHAPE == 0) {
                    const bool down = q[2] >= pl.bot;
                    const R zc = down ? pl.bot : pl.top;
                    x.lb = down ? L + 1 : L - 1;
                    const R th = (zc - y[F_Q + 2]) / (q[2] - y[F_Q + 2]);
                    x.th = (double)th;
                }
                break;
            }
            // no crossing after all (a last-bit difference to the listing kernel): the step stands
            s = layered_run<R, SHAPE>(M, fl, y, qc, dt, s, nsteps, true);
        }
        if (!hit) {
#pragma unroll
            for (int f = 0; f < NF; f++) st[(int64_t)f * cap + b] = y[f];
#pragma unroll
            for (int d = 0; d < 3; d++) st[(int64_t)(F_QC + d) * cap + b] = qc[d];
            continue;
        }
        const R head = (R)x.th * dt;
        straight_part<R>(S, head, y, qc);
#pragma unroll
        for (int f = 0; f < 18; f++) y[F_DQ + f] += head * B[f];
        double nrm[3] = {0.0, 0.0, 1.0};
        if (SHAPE == 0) {
            y[F_Q + 2] = x.lb > L ? pl.bot : pl.top;
            qc[2] = R(0);                 // the interface depth is exact
        } else {
            double p[3];
            for (int d = 0; d < 3; d++) p[d] = (double)y[F_Q + d] - (double)qc[d];
            if (SHAPE == 1) {
                double r[3], rn = 0.0;
                for (int d = 0; d < 3; d++) {
                    r[d] = p[d] - M.ctr[d];
                    rn += r[d] * r[d];
                }
                rn = sqrt(rn);
                for (int d = 0; d < 3; d++) {
                    nrm[d] = r[d] / rn;
                    p[d] = M.ctr[d] + x.rho * nrm[d];
                }
            } else {
                double h1, h2;
                p[2] = surf_at(M, x.iface, p[0], p[1], h1, h2);
                nrm[2] = rsqrt(1.0 + h1 * h1 + h2 * h2);
                nrm[0] = -h1 * nrm[2];
                nrm[1] = -h2 * nrm[2];
            }
            for (int d = 0; d < 3; d++) {
                y[F_Q + d] = (R)p[d];
                qc[d] = (R)((double)y[F_Q + d] - p[d]);
            }
        }
        EventOut ev;
        if (!interface_event<R, SHAPE>(M, fl, y, nrm, x.lb, rel_min, ev) || ev.n == 0) {
            flags[b] = fl | FL_DEAD;
            continue;
        }
        const long long pp = path[b];
        const int32_t id = ids[b];
        for (int k = 0; k < ev.n; k++) {
            R ch[NF], qch[3] = {qc[0], qc[1], qc[2]};
            make_child<R, SHAPE>(y, ev, nrm, k, ch);
            int flc = ev.flags[k];
            // the rest of the step, and the steps that follow
            const int sc = layered_run<R, SHAPE>(M, flc, ch, qch, dt, s + 1, nsteps, false, true,
                                                 SHAPE == 0 ? (R(1) - (R)x.th) * dt : R(1.0 - x.th) * dt);
            const bool again = sc < nsteps;
            if (again && ((flc >> 8) & 15) >= gmax) flc |= FL_DEAD;
            const int64_t dst = store_child<R>(st, flags, ids, path, cap, counts, b, k, ch, qch, flc, id, pp, ev.slot[k]);
            if (again && dst >= 0 && !(flc & FL_DEAD)) push_event(next, nnext, dst, sc);
        }
    }
}

fga_status launch_layered_steps(const fga_model *m, fga_beams *b, double dt, int nsteps, cudaStream_t s) {
    if (nsteps <= 0) return FGA_OK;
    // event lists: two of cap entries, and a counter per round (a lineage meets at most gmax interfaces, 16 by
    // its flag bits, and at most one per step)
    const int rounds = std::max(1, std::min(std::min(b->gmax, 16), nsteps));
    const size_t nb_ctr = sizeof(unsigned) * 20;
    // Where they do not fit (the device or the caller's bound): one shorter list.  The group is then taken step by step,
    // so that children meet no second interface in it, and slots entries of the population at a time.
    const int64_t cap = b->cap;
    int slots = (int)cap;
    FGA_TRY(ensure_scratch(b->events, slots, 1024, [&](int n) { return sizeof(int2) * (n == cap ? 2 : 1) * (size_t)n + nb_ctr; }));
    const bool whole = slots == cap;
    int2 *list[2] = {b->events.as<int2>(), b->events.as<int2>() + (whole ? cap : 0)};
    unsigned *ctr = reinterpret_cast<unsigned *>(b->events.as<char>() + sizeof(int2) * (whole ? 2 : 1) * (size_t)slots);
    auto go = [&](auto real, auto shape, int64_t first, int64_t end, int steps, int rounds) -> fga_status {
        using R = decltype(real);
        constexpr int SHAPE = decltype(shape)::value;
        unsigned long long *counts = b->counts.as<unsigned long long>();
        FGA_CUDA(cudaMemsetAsync(ctr, 0, nb_ctr, s));
        {
            ProfScope ps(P_PROP, s);
            layered_run_kernel<R, SHAPE><<<(unsigned)std::min<int64_t>((end - first + 127) / 128, 152 * 12), 128, 0, s>>>(
                m->dev, b->state.as<R>(), b->flags.as<int32_t>(), cap, counts, first, end, (R)dt, steps, b->gmax, list[0], ctr);
        }
        for (int r = 0; r < rounds; r++) {
            ProfScope ps(P_OTHER_LAYER, s);
            layered_event_kernel<R, SHAPE><<<152 * 8, 64, 0, s>>>(
                m->dev, b->state.as<R>(), b->flags.as<int32_t>(), b->id.as<int32_t>(), b->path.as<long long>(), cap,
                counts, (R)dt, steps, b->gmax, b->rel_min, list[r & 1], ctr + r, list[(r + 1) & 1], ctr + r + 1);
        }
        FGA_CUDA(cudaGetLastError());
        return FGA_OK;
    };
    auto run = [&](auto real, auto shape) -> fga_status {
        prof_add_beam_steps(b->nb * (int64_t)nsteps);
        if (whole) return go(real, shape, 0, cap, nsteps, rounds);
        for (int n = 0; n < nsteps; n++) {
            unsigned long long live = 0;   // the population of this step: children join at the next
            FGA_CUDA(cudaMemcpyAsync(&live, b->counts.p, sizeof live, cudaMemcpyDeviceToHost, s));
            FGA_CUDA(cudaStreamSynchronize(s));
            const int64_t nb = (int64_t)std::min<unsigned long long>(live, (unsigned long long)cap);
            for (int64_t first = 0; first < nb; first += slots)
                FGA_TRY(go(real, shape, first, std::min(first + slots, nb), 1, 1));
        }
        return FGA_OK;
    };
    using std::integral_constant;
    auto shape = [&](auto real) {
        return m->dev.shells  ? run(real, integral_constant<int, 1>{})
               : m->dev.undul ? run(real, integral_constant<int, 2>{})
                              : run(real, integral_constant<int, 0>{});
    };
    return b->precision == FGA_PREC_FP64 ? shape(double{}) : shape(float{});
}

}  // namespace fga
