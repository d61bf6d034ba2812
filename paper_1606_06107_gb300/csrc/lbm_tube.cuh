// The node update of the one-dimensional problems in float storage (D1Q7 +
// D1Q7): one node per thread (V = float: single steps and the many-step
// kernel, lbm_d1q7.cu) or two (V = F2: the ensemble, lbm_batch.cu).
//
// Every multiply-add is written out, no product feeds an addition directly
// (the packed instructions are contracted even where the scalar ones are not
// allowed to be; vmul_alone is the exception), and the files that include this
// are compiled without contraction, so each node's result is the same bits from
// either form.  Against the general kernel's expressions (k_step, contracted
// nowhere) the polynomial's coefficients are factored, mirror velocities share
// the equilibrium of h, the upwind stencil is three multiply-adds and the
// division by (D + n)/2 is a reciprocal product with one correction
// (Markstein, IBM J. Res. Dev. 34(1), 1990: correctly rounded, since 1/cT is):
// about 220 operations per node instead of 380 (1000 nodes, FD: 0.75 us per step
// in one launch, 1.04 with the general expressions).
//
// The order of the sums is part of the accuracy, because a rounding that recurs
// every step adds up over thousands of them: a new population is
// fma(1 - omega, old, small terms), so its own magnitude is rounded at once, and
// the second moment that corrects h^eq adds up the seven values one after
// another, as the general expressions do.  Error against the FP64 oracle over
// that of the general expressions, geometric mean of forty 1000-node FD tubes,
// n = 4, 2000 steps: rho 0.91, u 0.88, T 1.04 (tau 0.7-1), 0.82, 0.70, 1.08 (tau
// 2/3); 200 steps 0.95, 0.86, 0.97.  With fma(convection, .., fma(1 - omega, old,
// omega eq)) and half the moment doubled 1.69, 1.51, 2.08 and 1.69, 1.45, 2.85:
// 1-2 % faster in the ensemble.
#pragma once
#include "lbm_step.cuh"

namespace lbm {

__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float vmul(float a, float b) { return a * b; }
// a product that an addition follows, in a form that cannot be contracted
__device__ __forceinline__ float vmul_alone(float a, float b) { return a * b; }
__device__ __forceinline__ float vadd(float a, float b) { return a + b; }
__device__ __forceinline__ float vsub(float a, float b) { return a - b; }
__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ float vabs(float a) { return fabsf(a); }
__device__ __forceinline__ float vrcp(float a) { return __frcp_rn(a); }
__device__ __forceinline__ F2 vfma(F2 a, F2 b, F2 c) { return fma2(a, b, c); }
__device__ __forceinline__ F2 vmul(F2 a, F2 b) { return mul2(a, b); }
__device__ __forceinline__ F2 vmul_alone(F2 a, F2 b) { return f2(__fmul_rn(lo(a), lo(b)), __fmul_rn(hi(a), hi(b))); }
__device__ __forceinline__ F2 vadd(F2 a, F2 b) { return add2(a, b); }
__device__ __forceinline__ F2 vsub(F2 a, F2 b) { return sub2(a, b); }
__device__ __forceinline__ F2 vneg(F2 a) { return neg2(a); }
__device__ __forceinline__ F2 vabs(F2 a) { return F2{a.v & 0x7fffffff7fffffffull}; }
__device__ __forceinline__ F2 vrcp(F2 a) { return f2(__frcp_rn(lo(a)), __frcp_rn(hi(a))); }
template <typename V> struct Splat;
template <> struct Splat<float> {
    __device__ __forceinline__ static float of(float s) { return s; }
};
template <> struct Splat<F2> {
    __device__ __forceinline__ static F2 of(float s) { return f2(s); }
};

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

// One step of one node (or two).  ld(pop, d): population pop (g_0..g_6, then
// h_0..h_6) at node x + d.  stencil(ux) fixes the upwind side of h and
// returns a loader up(j, k): h_j two (k = 2) or one (1) nodes upwind, or one
// downwind (-1).  st(pop, v) stores.  rho and T are returned for the status.
template <bool ROT, int MODE, typename V, typename Ld, typename Stencil, typename St>
__device__ __forceinline__ void tube_update(const TubeLattice &c, const TubeRates &q, Ld &&ld, Stencil &&stencil,
                                            St &&st, V &rho_out, V &T_out)
{
    auto k1 = [](float s) { return Splat<V>::of(s); };
    V g[7], h[7];
#pragma unroll
    for (int i = 0; i < 7; ++i) g[i] = ld(i, MODE == 0 ? 3 - i : 0);
    if (ROT) {
#pragma unroll
        for (int j = 0; j < 7; ++j) h[j] = ld(7 + j, 0);
    }
    // ---- moments (Sec. V steps 3-4, Eq. T), opposite velocities first -------
    V rho = g[3], j = k1(0.f), e2 = k1(0.f), R2 = k1(0.f);
#pragma unroll
    for (int k = 1; k <= 3; ++k) {
        const V s = vadd(g[3 + k], g[3 - k]);
        rho = vadd(rho, s);
        j = vfma(k1((float)k), vsub(g[3 + k], g[3 - k]), j);
        e2 = vfma(k1((float)(k * k)), s, e2);
        if (ROT) R2 = vfma(k1((float)(k * k)), vadd(h[3 + k], h[3 - k]), R2);
    }
    const V inv_rho = vrcp(rho);
    const V ux = vmul(vmul(k1(c.r), j), inv_rho);
    const V j2 = vmul(j, j);
    V e = vmul(vmul(k1(0.5f), vfma(vneg(j2), inv_rho, e2)), inv_rho);
    if (ROT) e = vfma(k1(q.half_n), R2, e);
    // e / cT: the quotient's residual corrects the reciprocal product
    V T_lat = vmul(e, k1(q.inv_cT));
    T_lat = vfma(vfma(vneg(T_lat), k1(q.cT), e), k1(q.inv_cT), T_lat);
    const V E2_eq = vfma(rho, T_lat, vmul(j2, inv_rho));  // rho (u^2 + T) / r^2
    rho_out = rho;
    T_out = vmul(k1(c.r2), T_lat);

    // ---- coefficients of omega rho g^eq / w (eq_coef at D = 1) --------------
    const V t = vfma(k1(c.r2), T_lat, k1(-1.0f)), u2 = vmul(ux, ux), om = k1(q.omega), keep = k1(q.keep);
    const V scale = vmul(om, rho), st1 = vmul(scale, t);
    const V a00 = vmul(scale, vfma(u2, vfma(k1(0.75f), t, vfma(k1(0.125f), u2, k1(-0.5f))),
                                   vfma(t, vfma(k1(0.375f), t, k1(-0.5f)), k1(1.0f))));
    const V a01 = vmul(st1, vfma(k1(-0.75f), t, vfma(k1(-0.25f), u2, k1(0.5f))));
    const V a02 = vmul(k1(0.125f), vmul(st1, t));
    const V a10 = vmul(scale, vfma(k1(-1.5f), t, vfma(k1(-0.5f), u2, k1(1.0f))));
    const V a11 = vmul(k1(0.5f), st1);
    const V a20 = vmul(scale, vfma(k1(-1.25f), t, vfma(k1(-0.25f), u2, k1(0.5f))));
    const V a21 = vmul(k1(0.25f), st1);
    const V k6 = vmul(k1(1.0f / 6.0f), scale), k24 = vmul(k1(1.0f / 24.0f), scale);
    const V ru = vmul(k1(c.r), ux);

    // ---- collision and transport of g ---------------------------------------
    // the transport term of population i subtracted from v
    auto moved = [&](int i, V v) {
        if (MODE == 0) return v;
        const int ei = i - 3, m = ei < 0 ? -ei : ei, up = ei > 0 ? -1 : 1;
        if (m == 0) return v;
        V x = vfma(k1(-6.0f), ld(i, up), ld(i, 2 * up));
        x = vfma(k1(3.0f), g[i], x);
        x = vfma(k1(2.0f), ld(i, -up), x);
        return vfma(k1(-c.ce[m]), x, v);
    };
    V acc0 = k1(0.f), acc2 = k1(0.f), accj = k1(0.f), qm = k1(0.f), qp = k1(0.f);
#pragma unroll
    for (int m = 3; m >= 1; --m) {
        const V s = k1(c.s[m]), cu = vmul(k1((float)m), ru);
        const V A0 = vfma(s, vfma(s, a02, a01), a00), A1 = vfma(s, a11, a10), A2 = vfma(s, a21, a20);
        const V c2 = vmul(cu, cu);
        const V E = vfma(c2, vfma(c2, k24, A2), A0), O = vfma(c2, k6, A1);  // P(+-c) = E +- c O
        const V w = k1(c.w[m]);
        const V pp = vfma(cu, O, E), pm = vfma(vneg(cu), O, E), sum = vadd(pp, pm);
        acc0 = vfma(w, sum, acc0);
        acc2 = vfma(k1(c.w2[m]), sum, acc2);
        accj = vfma(k1(c.w1[m]), vsub(pp, pm), accj);
        if (m == 1) {  // stored last, with the corrections
            qm = pm;
            qp = pp;
        } else {
            st(3 - m, vfma(keep, g[3 - m], moved(3 - m, vmul(w, pm))));
            st(3 + m, vfma(keep, g[3 + m], moved(3 + m, vmul(w, pp))));
        }
    }
    acc0 = vfma(k1(c.w[0]), a00, acc0);
    const V d0 = vfma(om, rho, vneg(acc0));
    const V d2 = vfma(om, E2_eq, vneg(acc2));
    const V dm = vmul(k1(0.5f), vfma(om, j, vneg(accj)));
    st(3, vfma(keep, g[3], vfma(k1(c.w[0]), a00, vsub(d0, d2))));
    st(2, vfma(keep, g[2], moved(2, vfma(k1(c.w[1]), qm, vfma(k1(0.5f), d2, vneg(dm))))));
    st(4, vfma(keep, g[4], moved(4, vfma(k1(c.w[1]), qp, vfma(k1(0.5f), d2, dm)))));

    // ---- rotational populations ---------------------------------------------
    if (ROT) {
        // h^eq with its moments put right (heq_node): mirror entries are equal,
        // their contributions to the second moment still added one by one
        V eq[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) eq[k] = vfma(t, vfma(t, k1(c.hb[k]), k1(c.ha[k])), k1(1.0f));
        const V e1 = vmul_alone(k1(c.w[1]), eq[1]), e2w = vmul(k1(c.w[2]), eq[2]), e3 = vmul(k1(c.w[3]), eq[3]);
        V m2 = vfma(k1(4.0f), e2w, vmul(k1(9.0f), e3));
        m2 = vfma(k1(9.0f), e3, vfma(k1(4.0f), e2w, vadd(vadd(m2, e1), e1)));
        const V d = vsub(T_lat, m2);
        const V half0 = vadd(e1, vfma(k1(c.w[2]), eq[2], e3));
        eq[0] = vfma(k1(c.w[0]), eq[0], vsub(vfma(k1(-2.0f), half0, vfma(k1(-c.w[0]), eq[0], k1(1.0f))), d));
        eq[1] = vfma(k1(0.5f), d, e1);
        eq[2] = e2w;
        eq[3] = e3;
        const V anu = vneg(vabs(vmul(ux, k1(c.nu6))));
        auto up = stencil(ux);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
#pragma unroll
            for (int sgn = 0; sgn < (k ? 2 : 1); ++sgn) {
                const int jj7 = sgn ? 3 + k : 3 - k;
                V x = vfma(k1(-6.0f), up(jj7, 1), up(jj7, 2));
                x = vfma(k1(3.0f), h[jj7], x);
                x = vfma(k1(2.0f), up(jj7, -1), x);
                st(7 + jj7, vfma(keep, h[jj7], vfma(om, eq[k], vmul(anu, x))));
            }
        }
    }
}

__device__ __forceinline__ bool tube_bad(float rho, float T)
{
    return !(rho > 0.f) || !(T > 0.f) || !(fabsf(T) < 3.0e38f);
}

}  // namespace lbm
