// The node update of the one-dimensional problems in float storage (D1Q7 +
// D1Q7), one node per thread: single steps and the many-step kernel
// (lbm_d1q7.cu) and the ensemble (lbm_batch.cu).
//
// Every multiply-add is written out and the files that include this are
// compiled without contraction, so all of them give the same bits.  Against the
// general kernel's expressions (k_step) the polynomial's coefficients are
// factored, mirror velocities share the equilibrium of h, the upwind stencil is
// three multiply-adds and the division by (D + n)/2 is a reciprocal product with
// one correction (Markstein, IBM J. Res. Dev. 34(1), 1990: correctly rounded,
// since 1/cT is): about 220 operations per node instead of 380 (1000 nodes, FD:
// 0.75 us per step in one launch, 1.04 with the general expressions).
//
// The order of the sums is part of the accuracy, because a rounding that recurs
// every step adds up over thousands of them: a new population is
// fma(1 - omega, old, small terms), so its own magnitude is rounded at once, and
// the second moment that corrects h^eq adds up the seven values one after
// another, as the general expressions do.  Error against the FP64 oracle over
// that of the general expressions, geometric mean of forty 1000-node FD tubes,
// n = 4, 2000 steps: rho 0.91, u 0.88, T 1.04 (tau 0.7-1), 0.82, 0.70, 1.08 (tau
// 2/3); 200 steps 0.95, 0.86, 0.97.  With fma(convection, .., fma(1 - omega, old,
// omega eq)) and half the moment doubled 1.69, 1.51, 2.08 and 1.69, 1.45, 2.85.
#pragma once
#include "lbm_step.cuh"

namespace lbm {

// Constants of the lattice and the transport, by |e| = 0..3.
struct TubeLattice {
    float r, r2, nu6;  // nu6 = nu_scale / 6: u nu6 |stencil| is the convection term of h
    float w[4];        // translational and rotational weights (the same set)
    float w1[4], w2[4];  // w |e|, w e^2
    float s[4];        // r^2 e^2
    float ha[4], hb[4];  // h^eq_j / w_j = 1 + t ha + t^2 hb
    float ce[4];       // |e| / (6 m): finite-difference transport of g
};
inline TubeLattice tube_lattice(const float *w7, float r, float nu_scale, float inv_m)
{
    TubeLattice c{};
    c.r = r;
    c.r2 = r * r;
    c.nu6 = (float)((double)nu_scale / 6.0);
    for (int k = 0; k < 4; ++k) {
        c.w[k] = w7[3 + k];
        c.w1[k] = (float)((double)k * (double)c.w[k]);
        c.w2[k] = (float)((double)(k * k) * (double)c.w[k]);
        c.s[k] = c.r2 * (float)(k * k);
        const double s = c.s[k];
        c.ha[k] = (float)(0.5 * (s - 1.0));
        c.hb[k] = (float)(0.125 * (s * s - 6.0 * s + 3.0));
        c.ce[k] = (float)((double)k * (double)inv_m / 6.0);
    }
    return c;
}

// Constants of one problem.
struct TubeRates {
    float omega, keep;   // keep = 1 - omega, exact
    float cT, inv_cT;    // (D + n) / 2 and its correctly rounded reciprocal
    float half_n;
};
__host__ __device__ __forceinline__ TubeRates tube_rates(float omega, float cT, float half_n)
{
    return TubeRates{omega, 1.0f - omega, cT, 1.0f / cT, half_n};
}

// One step of one node.  ld(pop, d): population pop (g_0..g_6, then h_0..h_6)
// at node x + d.  stencil(ux) fixes the upwind side of h and returns a loader
// up(j, k): h_j two (k = 2) or one (1) nodes upwind, or one downwind (-1).  The
// new populations come back in `out`, for the caller to store together (a load
// does not move above a store that might be to the same address); rho and T
// are returned for the status.
template <bool ROT, int MODE, typename Ld, typename Stencil>
__device__ __forceinline__ void tube_update(const TubeLattice &c, const TubeRates &q, Ld &&ld, Stencil &&stencil,
                                            float (&out)[ROT ? 14 : 7], float &rho_out, float &T_out)
{
    float g[7], h[7];
#pragma unroll
    for (int i = 0; i < 7; ++i) g[i] = ld(i, MODE == 0 ? 3 - i : 0);
    if (ROT) {
#pragma unroll
        for (int j = 0; j < 7; ++j) h[j] = ld(7 + j, 0);
    }
    // ---- moments (Sec. V steps 3-4, Eq. T), opposite velocities first -------
    float rho = g[3], j = 0.f, e2 = 0.f, R2 = 0.f;
#pragma unroll
    for (int k = 1; k <= 3; ++k) {
        const float s = g[3 + k] + g[3 - k];
        rho += s;
        j = fmaf((float)k, g[3 + k] - g[3 - k], j);
        e2 = fmaf((float)(k * k), s, e2);
        if (ROT) R2 = fmaf((float)(k * k), h[3 + k] + h[3 - k], R2);
    }
    const float inv_rho = __frcp_rn(rho);
    const float ux = c.r * j * inv_rho, j2 = j * j;
    float e = 0.5f * fmaf(-j2, inv_rho, e2) * inv_rho;
    if (ROT) e = fmaf(q.half_n, R2, e);
    // e / cT: the quotient's residual corrects the reciprocal product
    float T_lat = e * q.inv_cT;
    T_lat = fmaf(fmaf(-T_lat, q.cT, e), q.inv_cT, T_lat);
    const float E2_eq = fmaf(rho, T_lat, j2 * inv_rho);  // rho (u^2 + T) / r^2
    rho_out = rho;
    T_out = c.r2 * T_lat;

    // ---- coefficients of omega rho g^eq / w (eq_coef at D = 1) --------------
    const float t = fmaf(c.r2, T_lat, -1.0f), u2 = ux * ux, om = q.omega, keep = q.keep;
    const float scale = om * rho, st = scale * t;
    const float a00 = scale * fmaf(u2, fmaf(0.75f, t, fmaf(0.125f, u2, -0.5f)), fmaf(t, fmaf(0.375f, t, -0.5f), 1.0f));
    const float a01 = st * fmaf(-0.75f, t, fmaf(-0.25f, u2, 0.5f)), a02 = 0.125f * (st * t);
    const float a10 = scale * fmaf(-1.5f, t, fmaf(-0.5f, u2, 1.0f)), a11 = 0.5f * st;
    const float a20 = scale * fmaf(-1.25f, t, fmaf(-0.25f, u2, 0.5f)), a21 = 0.25f * st;
    const float k6 = (1.0f / 6.0f) * scale, k24 = (1.0f / 24.0f) * scale;
    const float ru = c.r * ux;

    // ---- collision and transport of g ---------------------------------------
    // (1 - omega) g_i + v less the transport term
    auto put = [&](int i, float v) {
        const int ei = i - 3, m = ei < 0 ? -ei : ei, up = ei > 0 ? -1 : 1;
        if (MODE == 1 && m != 0) {
            float x = fmaf(-6.0f, ld(i, up), ld(i, 2 * up));
            x = fmaf(3.0f, g[i], x);
            x = fmaf(2.0f, ld(i, -up), x);
            v = fmaf(-c.ce[m], x, v);
        }
        out[i] = fmaf(keep, g[i], v);
    };
    float acc0 = 0.f, acc2 = 0.f, accj = 0.f, qm = 0.f, qp = 0.f;
#pragma unroll
    for (int m = 3; m >= 1; --m) {
        const float s = c.s[m], cu = (float)m * ru, c2 = cu * cu;
        const float A0 = fmaf(s, fmaf(s, a02, a01), a00), A1 = fmaf(s, a11, a10), A2 = fmaf(s, a21, a20);
        const float E = fmaf(c2, fmaf(c2, k24, A2), A0), O = fmaf(c2, k6, A1);  // P(+-c) = E +- c O
        const float w = c.w[m], pp = fmaf(cu, O, E), pm = fmaf(-cu, O, E), sum = pp + pm;
        acc0 = fmaf(w, sum, acc0);
        acc2 = fmaf(c.w2[m], sum, acc2);
        accj = fmaf(c.w1[m], pp - pm, accj);
        if (m == 1) {  // last, with the corrections
            qm = pm;
            qp = pp;
        } else {
            put(3 - m, w * pm);
            put(3 + m, w * pp);
        }
    }
    acc0 = fmaf(c.w[0], a00, acc0);
    const float d0 = fmaf(om, rho, -acc0);
    const float d2 = fmaf(om, E2_eq, -acc2);
    const float dm = 0.5f * fmaf(om, j, -accj);
    put(3, fmaf(c.w[0], a00, d0 - d2));
    put(2, fmaf(c.w[1], qm, fmaf(0.5f, d2, -dm)));
    put(4, fmaf(c.w[1], qp, fmaf(0.5f, d2, dm)));

    // ---- rotational populations ---------------------------------------------
    if (ROT) {
        // h^eq with its moments put right (heq_node): mirror entries are equal,
        // their contributions to the second moment still added one by one
        float eq[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) eq[k] = fmaf(t, fmaf(t, c.hb[k], c.ha[k]), 1.0f);
        const float q1 = c.w[1] * eq[1], q2 = c.w[2] * eq[2], q3 = c.w[3] * eq[3];
        const float m2 = fmaf(9.0f, q3, fmaf(4.0f, q2, fmaf(4.0f, q2, 9.0f * q3) + q1 + q1));
        const float d = T_lat - m2;
        const float half0 = q1 + fmaf(c.w[2], eq[2], q3);
        eq[0] = fmaf(c.w[0], eq[0], fmaf(-2.0f, half0, fmaf(-c.w[0], eq[0], 1.0f)) - d);
        eq[1] = fmaf(0.5f, d, q1);
        eq[2] = q2;
        eq[3] = q3;
        const float anu = -fabsf(ux * c.nu6);
        auto up = stencil(ux);
#pragma unroll
        for (int j7 = 0; j7 < 7; ++j7) {
            float x = fmaf(-6.0f, up(j7, 1), up(j7, 2));
            x = fmaf(3.0f, h[j7], x);
            x = fmaf(2.0f, up(j7, -1), x);
            out[7 + j7] = fmaf(keep, h[j7], fmaf(om, eq[j7 < 3 ? 3 - j7 : j7 - 3], anu * x));
        }
    }
}

__device__ __forceinline__ bool tube_bad(float rho, float T)
{
    return !(rho > 0.f) || !(T > 0.f) || !(fabsf(T) < 3.0e38f);
}

}  // namespace lbm
