// Beams where the speed is constant (constant media, the inside of a homogeneous layer).  With grad c = 0
// the ODEs of Eqs. char_plus/minus, DzDt, amp_* reduce to
//   Q' = sg c P^,  P' = 0,  dzQ' = B = sg (c/|P|) (dzP - (dzP P^) P^T),  dzP' = 0,
//   a' = gamma a,  gamma = tr(Z^-1 B)/2,  Z(t) = Z(0) + t B        (no SV/SH coupling: P is constant)
// with constant slopes of Q and dzQ, on which a classical RK4 step is exact, and det Z(t) = det Z(0)
// (1 + e1 t + e2 t^2) because B P^ = 0 (det B = 0).  So gamma = (e1 + 2 e2 t)/(1 + e1 t + e2 t^2)/2 at every
// stage of every step follows from two complex numbers per beam, and the RK4 step of a is a complex factor
// formed from gamma at its start, middle and end: the same discrete map as four evaluations of the general
// right-hand side, for about 80 floating-point operations per step instead of 4,200.
#pragma once

#include "fga_beam.cuh"

namespace fga {

// steps after which the expansion of det Z is renewed at the current state
constexpr int STRAIGHT_RENEW = 64;

template <typename R> struct Straight {
    R v[3];          // Q'
    C2<R> e1, e2;    // det Z(t) / det Z(0) = 1 + e1 t + e2 t^2
};

// B (18 reals, ordered as dzQ in the state) and the expansion of a beam state
template <typename R>
__device__ __forceinline__ void straight_setup(R sg, R c, const R *y, R *B, Straight<R> &S) {
    const R P[3] = {y[F_P], y[F_P + 1], y[F_P + 2]};
    const R ip = Real<R>::rsqrt_(P[0] * P[0] + P[1] * P[1] + P[2] * P[2]);
    const R Ph[3] = {P[0] * ip, P[1] * ip, P[2] * ip};
    const R sc = sg * c, scip = sg * (c * ip);
#pragma unroll
    for (int d = 0; d < 3; d++) S.v[d] = sc * Ph[d];
    C2<R> Z[3][3], Z1[3][3], Cf[3][3];
#pragma unroll
    for (int m = 0; m < 3; m++) {
        R vr = R(0), vi = R(0);
#pragma unroll
        for (int l = 0; l < 3; l++) {
            vr += y[F_DP + 2 * (3 * m + l)] * Ph[l];
            vi += y[F_DP + 2 * (3 * m + l) + 1] * Ph[l];
        }
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const int e = 2 * (3 * m + j);
            B[e] = scip * (y[F_DP + e] - vr * Ph[j]);
            B[e + 1] = scip * (y[F_DP + e + 1] - vi * Ph[j]);
            Z[m][j] = {y[F_DQ + e] - y[F_DP + e + 1], y[F_DQ + e + 1] + y[F_DP + e]};
            Z1[m][j] = {B[e], B[e + 1]};
        }
    }
    auto cof = [&](C2<R> (&M)[3][3]) {
#pragma unroll
        for (int m = 0; m < 3; m++) {
            const int a = (m + 1) % 3, b = (m + 2) % 3;
#pragma unroll
            for (int j = 0; j < 3; j++) {
                const int p = (j + 1) % 3, q = (j + 2) % 3;
                Cf[m][j] = cmulsub(M[a][p], M[b][q], M[a][q], M[b][p]);
            }
        }
    };
    auto dot = [&](C2<R> (&M)[3][3], int rows) {
        C2<R> s = {R(0), R(0)};
#pragma unroll
        for (int m = 0; m < 3; m++)
            if (m < rows)
#pragma unroll
                for (int j = 0; j < 3; j++) {
                    const C2<R> t = cmul(Cf[m][j], M[m][j]);
                    s.r += t.r;
                    s.i += t.i;
                }
        return s;
    };
    cof(Z);
    const C2<R> d0 = dot(Z, 1), d1 = dot(Z1, 3);
    cof(Z1);
    const C2<R> d2 = dot(Z, 3);
    // 1/d0 with |d0| scaled to 1 first (the Jacobian of a beam refracted near grazing is large)
    const R big = fmax(fabs(d0.r), fabs(d0.i)), sc0 = R(1) / big;
    const R ur = d0.r * sc0, ui = d0.i * sc0, in = sc0 / (ur * ur + ui * ui);
    const C2<R> id = {ur * in, -ui * in};
    S.e1 = cmul(d1, id);
    S.e2 = cmul(d2, id);
}

// gamma at time t after the expansion
template <typename R> __device__ __forceinline__ C2<R> straight_gamma(const Straight<R> &S, R t) {
    const R pr = R(1) + t * (S.e1.r + t * S.e2.r), pi = t * (S.e1.i + t * S.e2.i);
    const R qr = S.e1.r + R(2) * t * S.e2.r, qi = S.e1.i + R(2) * t * S.e2.i;
    const R in = R(0.5) * Real<R>::rcp_pos_(pr * pr + pi * pi);
    return {(qr * pr + qi * pi) * in, (qi * pr - qr * pi) * in};
}

// gamma at two times; in FP64 with one division for both (a division is some ten operations of the FP64 pipe)
template <typename R>
__device__ __forceinline__ void straight_gamma2(const Straight<R> &S, R ta, R tb, C2<R> &ga, C2<R> &gb) {
    if (sizeof(R) == 4) {
        ga = straight_gamma<R>(S, ta);
        gb = straight_gamma<R>(S, tb);
        return;
    }
    const R ar = R(1) + ta * (S.e1.r + ta * S.e2.r), ai = ta * (S.e1.i + ta * S.e2.i);
    const R br = R(1) + tb * (S.e1.r + tb * S.e2.r), bi = tb * (S.e1.i + tb * S.e2.i);
    const R ta2 = R(2) * ta, tb2 = R(2) * tb;
    const R pr = S.e1.r + ta2 * S.e2.r, pi = S.e1.i + ta2 * S.e2.i, qr = S.e1.r + tb2 * S.e2.r, qi = S.e1.i + tb2 * S.e2.i;
    const R na = ar * ar + ai * ai, nb = br * br + bi * bi, in = R(0.5) / (na * nb), ia = in * nb, ib = in * na;
    ga = {(pr * ar + pi * ai) * ia, (pi * ar - pr * ai) * ia};
    gb = {(qr * br + qi * bi) * ib, (qi * br - qr * bi) * ib};
}

// the relative increment of a over one RK4 step h from gamma at its start, middle and end
template <typename R> __device__ __forceinline__ C2<R> straight_gain(R h, C2<R> g1, C2<R> g2, C2<R> g4) {
    const R hh = R(0.5) * h;
    const C2<R> k2 = cmul(g2, C2<R>{R(1) + hh * g1.r, hh * g1.i});
    const C2<R> k3 = cmul(g2, C2<R>{R(1) + hh * k2.r, hh * k2.i});
    const C2<R> k4 = cmul(g4, C2<R>{R(1) + h * k3.r, h * k3.i});
    const R h6 = h / R(6);
    return {h6 * (g1.r + R(2) * (k2.r + k3.r) + k4.r), h6 * (g1.i + R(2) * (k2.i + k3.i) + k4.i)};
}

template <typename R> __device__ __forceinline__ void straight_amplitudes(R *y, C2<R> g) {
#pragma unroll
    for (int f = F_A0; f < NF; f += 2) {
        const R ar = y[f], ai = y[f + 1];
        y[f] = ar + (g.r * ar - g.i * ai);
        y[f + 1] = ai + (g.r * ai + g.i * ar);
    }
}

// Q by compensated summation over a step h
template <typename R> __device__ __forceinline__ void straight_q(const Straight<R> &S, R h, R *q, R *qc) {
#pragma unroll
    for (int d = 0; d < 3; d++) kahan_add<R>(q[d], qc[d], h * S.v[d]);
}

// Q and the amplitudes over a step h from the expansion's start (dzQ += h B is the caller's)
template <typename R> __device__ __forceinline__ void straight_part(const Straight<R> &S, R h, R *y, R *qc) {
    straight_amplitudes<R>(y, straight_gain<R>(h, straight_gamma<R>(S, R(0)), straight_gamma<R>(S, R(0.5) * h),
                                               straight_gamma<R>(S, h)));
    straight_q<R>(S, h, y + F_Q, qc);
}

}  // namespace fga
