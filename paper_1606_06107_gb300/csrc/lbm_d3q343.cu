// Kernel instantiations for the D3Q343 lattice (D1Q7 x D1Q7 x D1Q7) and its
// two-pass STREAM step.
//
// 343 populations do not fit in registers, so the step reads its pulled
// populations twice: a first pass accumulates rho, j and sum |e|^2 g (row
// sums by (e_y, e_z), column sums by e_x), a second pass re-reads each value
// (from a shared-memory stash for the first planes with 16-bit storage, else
// from L1/L2: a 128-node block touches 343 x 128 x 4 B = 175 KB between the
// two reads) and writes its post-collision value (with 16-bit storage as a
// deviation computed from the stored deviation, two nodes per thread, below).
// The second pass walks the e_z planes in reverse, so that it starts on the
// lines the first pass loaded last, which are the ones still in L1 (7 % faster
// with float storage).  The rest and the six unit velocities are stored last
// with the float32 moment corrections, as in the one- and two-dimensional
// kernels.  Element indices are 64-bit (the state of a 384^3 grid holds
// 2 x 10^10 values).
#include "lbm_step.cuh"

namespace lbm {
namespace {

constexpr int kQ343 = 343;

// Float storage: resident blocks per SM the register allocation must allow
// and threads per block (x positions of one row).  Left free the compiler
// takes 185-207 registers (2 blocks of 4 warps); 3 blocks measured 13 % (n =
// 0) and 7 % (n = 4) faster.  Narrower blocks share fewer of the pulled rows'
// lines in L1.
#ifndef LBM_Q343_MIN_BLOCKS
#define LBM_Q343_MIN_BLOCKS 3
#endif
constexpr int kQ343Block = 128;

// Population i of the node at in-population offset off (64-bit element
// index: the state of a 384^3 grid holds 2 x 10^10 values).
__device__ __forceinline__ float q343_load(const Params<kQ343> &p, int i, int off)
{
    return ld_ro(p.src + ((uint64_t)i * (uint64_t)p.S + (uint64_t)(uint32_t)off));
}
__device__ __forceinline__ void q343_store(const Params<kQ343> &p, int i, int self, float v)
{
    p.dst[(uint64_t)i * (uint64_t)p.S + (uint32_t)self] = v;
}

// Pass 2 with 16-bit deviation storage, d_i = f_i / w_i - 1, runs on the
// deviations with the weights factored.  D3Q343 = D1Q7^3, so w_i = w_a w_b
// w_c.  The e_z planes c are a run-time loop, so a table lookup w[i] (or
// 1 / w[i]) is a run-time-indexed parameter load for every population; here
// the in-plane factors w_a w_b, w_a w_b e_x and w_a w_b e_x^2 (compile-time
// indices inside the unrolled row) are immediate operands of the row sums and
// the plane factor w_c multiplies the plane sums once.  The collision
// f* = (1 - omega) g + omega g^eq becomes d* = (1 - omega) d + (P - omega)
// with P = omega rho g^eq / w, so no value is decoded to f or encoded back.
// The equilibrium along each row is evaluated as a quartic in e_x (below),
// 6 operations per pair of populations e_x = +-k instead of a full
// polynomial evaluation for each.  (With the weight table and a polynomial
// per population pass 2 took 20 % longer; the same treatment of pass 1 cost
// registers and gained nothing.)
struct Q343Weights {
    float w2[49];    // w_a w_b, index b * 7 + a
    float w2x[49];   // w_a w_b e_x
    float w2x2[49];  // w_a w_b e_x^2
    float wc[7];     // w_c
    float iw_rest, iw_unit;  // 1 / w of the rest velocity and of the unit velocities
};
// The five sums of pass 1: rho, j and sum_i |e_i|^2 g_i (lattice units).
struct Q343Sums {
    float rho, jx, jy, jz, e2;
};

// Pass 1 of one node: moments of the pulled populations g_i(x) = ft_i(x - e_i).
__device__ __forceinline__ Q343Sums q343_sums(const Params<kQ343> &p, const Offsets &o, int z)
{
    const int plane = p.pitch * p.Y;
    float cs[7];
#pragma unroll
    for (int a = 0; a < 7; ++a) cs[a] = 0.f;
    float rho = 0.f, jy = 0.f, jz = 0.f, e2yz = 0.f;
    // e_y is unrolled so that each e_z plane issues its 49 loads at once
    for (int c = 0; c < 7; ++c) {
        const int zo = bc_wrap(z - (c - 3), p.Z, p.bc2) * plane;
#pragma unroll
        for (int b = 0; b < 7; ++b) {
            const int row = zo + o.y[6 - b];
            float rsum = 0.f;
#pragma unroll
            for (int a = 0; a < 7; ++a) {
                const float g = q343_load(p, (c * 7 + b) * 7 + a, row + o.x[6 - a]);
                cs[a] += g;
                rsum += g;
            }
            const float db = (float)(b - 3), dc = (float)(c - 3);
            rho += rsum;
            jy = fmaf(db, rsum, jy);
            jz = fmaf(dc, rsum, jz);
            e2yz = fmaf(db * db + dc * dc, rsum, e2yz);
        }
    }
    float jx = 0.f, e2 = e2yz;
#pragma unroll
    for (int k = 1; k <= 3; ++k) {
        jx = fmaf((float)k, cs[3 + k] - cs[3 - k], jx);
        e2 = fmaf((float)(k * k), cs[3 + k] + cs[3 - k], e2);
    }
    return Q343Sums{rho, jx, jy, jz, e2};
}

// The equilibrium polynomial along a row.  With e_y, e_z fixed, c = xi . u
// = C0 + e_x v and s = |xi|^2 = S0 + r^2 e_x^2, so P = A0(s) + A1(s) c +
// A2(s) c^2 + k6 c^3 + k24 c^4 (eq_single) is a quartic in e_x, b0 + b1 e_x
// + b2 e_x^2 + b3 e_x^3 + b4 e_x^4, with b0 = P(C0, S0), b1 = v dP/dc and
// b2, b3 from expanding it; b4 is the same for every row.  The pairs
// e_x = +-k share the even part b0 + b2 k^2 + b4 k^4 and the odd part
// k (b1 + b3 k^2): about 25 operations per row and 6 per pair.
struct RowQuartic {
    float v, v2, k3k6, k4k24, k6k24, a02x2, a21x2, b4;
};
__device__ __forceinline__ RowQuartic row_quartic_setup(const EqCoef &k, float v, float r2)
{
    RowQuartic q;
    q.v = v;
    q.v2 = v * v;
    q.k3k6 = 3.0f * k.k6;
    q.k4k24 = 4.0f * k.k24;
    q.k6k24 = 6.0f * k.k24;
    q.a02x2 = 2.0f * k.a02;
    q.a21x2 = 2.0f * k.a21;
    q.b4 = fmaf(k.a02, r2 * r2, fmaf(k.a21 * r2, q.v2, k.k24 * q.v2 * q.v2));
    return q;
}
// P at e_x = a - 3, a = 0..6, of the row with c = C0 + e_x v, s = S0 + r2 e_x^2.
__device__ __forceinline__ void row_quartic(const EqCoef &k, const RowQuartic &q, float r2, float C0, float S0,
                                            float (&P)[7])
{
    const float A0 = fmaf(S0, fmaf(S0, k.a02, k.a01), k.a00);
    const float A1 = fmaf(S0, k.a11, k.a10);
    const float A2 = fmaf(S0, k.a21, k.a20);
    const float b0 = fmaf(C0, fmaf(C0, fmaf(C0, fmaf(C0, k.k24, k.k6), A2), A1), A0);
    const float b1 = q.v * fmaf(C0, fmaf(C0, fmaf(C0, q.k4k24, q.k3k6), A2 + A2), A1);
    const float b2 = fmaf(r2, fmaf(C0, fmaf(C0, k.a21, k.a11), fmaf(q.a02x2, S0, k.a01)),
                          q.v2 * fmaf(C0, fmaf(C0, q.k6k24, q.k3k6), A2));
    const float b3 = q.v * fmaf(r2, fmaf(C0, q.a21x2, k.a11), q.v2 * fmaf(C0, q.k4k24, k.k6));
    P[3] = b0;
#pragma unroll
    for (int m = 1; m <= 3; ++m) {
        const float E = fmaf(q.b4, (float)(m * m * m * m), fmaf(b2, (float)(m * m), b0));
        const float O = (float)m * fmaf(b3, (float)(m * m), b1);
        P[3 + m] = E + O;
        P[3 - m] = E - O;
    }
}

// Pass 2 of one node and the rotational update: moments, equilibrium, BGK,
// store (the rest and the unit velocities deferred).  Each q_i = w_i P_i with
// P from the row quartic and w_i = (w_a w_b) w_c (an immediate times the
// plane's factor); the correction sums run over the q_i that are stored.
// Float storage: 10.4 ms per step on a 256^3 blast (n = 0) against 10.6 with
// the weight table and a polynomial per population.
template <bool ROT>
__device__ __forceinline__ void q343_collide(const Params<kQ343> &p, const Q343Weights &qw, const Offsets &o, int z,
                                             const Q343Sums &s)
{
    constexpr int D = 3;
    constexpr int C = (kQ343 - 1) / 2;  // rest velocity (171)
    const int plane = p.pitch * p.Y;
    float h[7], R2 = 0.f;
    if (ROT) {
#pragma unroll
        for (int j = 0; j < 7; ++j) h[j] = ld(p, kQ343 + j, o.self());
#pragma unroll
        for (int k = 1; k <= 3; ++k) R2 = fmaf((float)(k * k), h[3 + k] + h[3 - k], R2);
    }
    const Moments m = make_moments<D, ROT>(p, s.rho, s.jx, s.jy, s.jz, s.e2, R2);
    if (!(m.rho > 0.f) || !(m.T > 0.f) || !(fabsf(m.T) < 3.0e38f)) atomicOr(p.status, 1);

    const float u2 = m.ux * m.ux + m.uy * m.uy + m.uz * m.uz;
    const float om_rho = p.omega * m.rho;
    const EqCoef k = eq_coef<D>(m.T, u2, om_rho);  // omega rho g^eq / w_i
    const float keep = 1.0f - p.omega;
    const float rux = m.ux * p.r, ruy = m.uy * p.r, ruz = m.uz * p.r;
    const int self = o.self();
    const RowQuartic rq = row_quartic_setup(k, rux, p.r2);
    float acc0 = 0.f, acc2 = 0.f, ax = 0.f, ay = 0.f, az = 0.f;
    float q_c = 0.f, q_mx = 0.f, q_px = 0.f, q_my = 0.f, q_py = 0.f, q_mz = 0.f, q_pz = 0.f;
    float g_c = 0.f, g_mx = 0.f, g_px = 0.f, g_my = 0.f, g_py = 0.f, g_mz = 0.f, g_pz = 0.f;
    // The correction sums are accumulated per row of 7 and then per plane, so
    // each carries the rounding of ~2 x 7 additions rather than of 343.
    // Planes in reverse order (see above).
    for (int c = 6; c >= 0; --c) {
        const int zo = bc_wrap(z - (c - 3), p.Z, p.bc2) * plane;
        const int ez = c - 3;
        const float wc = qw.wc[c];
        float p0 = 0.f, p2 = 0.f, px = 0.f, py = 0.f;  // plane sums
#pragma unroll
        for (int b = 0; b < 7; ++b) {
            const int row = zo + o.y[6 - b];
            const int ey = b - 3;
            const float cyz = fmaf((float)ey, ruy, (float)ez * ruz);
            const int e2yz_i = ey * ey + ez * ez;
            const float eyz2 = (float)e2yz_i;
            float Prow[7];
            row_quartic(k, rq, p.r2, cyz, p.r2 * eyz2, Prow);
            float r0 = 0.f, r2 = 0.f, rx = 0.f;  // row sums
#pragma unroll
            for (int a = 0; a < 7; ++a) {
                const int ex = a - 3;
                const int i = (c * 7 + b) * 7 + a;
                const int E2 = ex * ex + e2yz_i;
                const float q = (qw.w2[b * 7 + a] * wc) * Prow[a];  // w_i = (w_a w_b) w_c
                r0 += q;
                if (ex) {
                    r2 = fmaf((float)(ex * ex), q, r2);
                    rx = fmaf((float)ex, q, rx);
                }
                const float g = q343_load(p, i, row + o.x[6 - a]);
                if (E2 <= 1) {  // the rest and the six unit velocities: stored last
                    if (E2 == 0) { q_c = q; g_c = g; }
                    else if (ex == -1) { q_mx = q; g_mx = g; }
                    else if (ex == 1) { q_px = q; g_px = g; }
                    else if (ey == -1) { q_my = q; g_my = g; }
                    else if (ey == 1) { q_py = q; g_py = g; }
                    else if (ez == -1) { q_mz = q; g_mz = g; }
                    else { q_pz = q; g_pz = g; }
                } else {
                    q343_store(p, i, self, fmaf(keep, g, q));
                }
            }
            p0 += r0;
            p2 += fmaf(eyz2, r0, r2);
            px += rx;
            py = fmaf((float)ey, r0, py);
        }
        acc0 += p0;
        acc2 += p2;
        ax += px;
        ay += py;
        az = fmaf((float)ez, p0, az);
    }
    const float d0 = om_rho - acc0;
    const float d2 = p.omega * m.E2_eq - acc2;
    const float bb = d2 * (0.5f / (float)D);
    const float dmx = 0.5f * (p.omega * m.j[0] - ax);
    const float dmy = 0.5f * (p.omega * m.j[1] - ay);
    const float dmz = 0.5f * (p.omega * m.j[2] - az);
    q343_store(p, C, self, fmaf(keep, g_c, q_c + (d0 - d2)));
    q343_store(p, C - 1, self, fmaf(keep, g_mx, q_mx + (bb - dmx)));
    q343_store(p, C + 1, self, fmaf(keep, g_px, q_px + (bb + dmx)));
    q343_store(p, C - 7, self, fmaf(keep, g_my, q_my + (bb - dmy)));
    q343_store(p, C + 7, self, fmaf(keep, g_py, q_py + (bb + dmy)));
    q343_store(p, C - 49, self, fmaf(keep, g_mz, q_mz + (bb - dmz)));
    q343_store(p, C + 49, self, fmaf(keep, g_pz, q_pz + (bb + dmz)));

    if (ROT) {
        float adv[7];
        rot_advect<D>(p, o, h, m, adv);
        rot_store(p, self, h, m, adv);
    }
}

// ---------------------------------------------------------------------------
// 16-bit storage: the same two passes on two x-adjacent nodes per thread
// (lbm_step_pair.cuh: packed arithmetic, 32-bit loads, stash entries and
// stores).  Pass 1 keeps the raw pairs of the e_z planes c < kPairStash in
// shared memory for pass 2, which reaches them last, when L1 has long evicted
// them; it works on the same stored bits, so the depth does not change
// results.  Bound by load latency and issue at the resident warps (255
// registers: eight warps an SM).  256^3 half, n = 0 / n = 4, ms per step, by
// threads per block, stash planes and resident blocks per SM: 64, 4, 4: 7.69 /
// 8.60 (kept); 64, 5, 3: 8.11 / 9.48; 64, 6, 3: 9.35 / 9.96; 64, 3, 6: 8.82 /
// 9.46; 128, 3, 3: 7.75 / 8.55; 128, 0, 3: 8.41 / 9.71; 32, 4, 8: 8.33 / 9.36; one
// node per thread (128, 6, 3): 8.22 / 9.48.
//
// A block is part of a row, so rows of an odd number of warps (2 x 32 nodes each)
// take blocks of one warp: in blocks of two the last warp has no nodes and keeps
// its registers.  us per step, n = 4, in blocks of 32 / 64: 36 x 36 x 25 33 / 54 (47
// with one node per thread), 64 x 60 x 58 119 / 207 (190), 131 x 128 x 120 1718 /
// 2068 (2547); even rows 78 x 82 x 72 415 / 371, 128^3 1118 / 975.
#ifndef LBM_Q343_PAIR_STASH
#define LBM_Q343_PAIR_STASH 4
#endif
constexpr int kPairWarps = 8;  // resident warps per SM that the registers allow
constexpr int kPairStash = LBM_Q343_PAIR_STASH;
template <int BLOCK> constexpr size_t pair_stash_bytes() { return (size_t)kPairStash * 49 * BLOCK * 4; }

struct Q343PairSums {
    F2 rho, jx, jy, jz, e2;
};

// q343_sums of both nodes.
template <int NS, int BLOCK, bool WHOLE, typename ST>
__device__ __forceinline__ Q343PairSums q343_pair_sums(const Params<kQ343, ST> &p, const PairOffsets &o, int z,
                                                       uint32_t *stash)
{
    const int plane = p.pitch * p.Y;
    F2 cs[7];
#pragma unroll
    for (int a = 0; a < 7; ++a) cs[a] = f2(0.f);
    F2 rho = f2(0.f), jy = f2(0.f), jz = f2(0.f), e2yz = f2(0.f);
    auto plane1 = [&](auto keep, int c) {
        constexpr bool KEEP = decltype(keep)::value;
        const int zo = bc_wrap(z - (c - 3), p.Z, p.bc2) * plane;
#pragma unroll
        for (int b = 0; b < 7; ++b) {
            const int row = zo + o.y[6 - b];
            F2 rsum = f2(0.f);
#pragma unroll
            for (int a = 0; a < 7; ++a) {
                const int i = (c * 7 + b) * 7 + a;
                const uint32_t v = ld_pair<WHOLE>(p, i, row, o, 3 - a);
                if constexpr (KEEP) stash[i * BLOCK + threadIdx.x] = v;
                const F2 w = f2(p.w[i]);
                const F2 g = fma2(w, Pair16<ST>::get(v), w);
                cs[a] = add2(cs[a], g);
                rsum = a ? add2(rsum, g) : g;
            }
            const float db = (float)(b - 3), dc = (float)(c - 3);
            rho = add2(rho, rsum);
            jy = fma2(f2(db), rsum, jy);
            jz = fma2(f2(dc), rsum, jz);
            e2yz = fma2(f2(db * db + dc * dc), rsum, e2yz);
        }
    };
#pragma unroll 1
    for (int c = 0; c < 7; ++c) {
        if (c < NS) plane1(std::true_type{}, c);
        else plane1(std::false_type{}, c);
    }
    F2 jx = f2(0.f), e2 = e2yz;
#pragma unroll
    for (int k = 1; k <= 3; ++k) {
        jx = fma2(f2((float)k), sub2(cs[3 + k], cs[3 - k]), jx);
        e2 = fma2(f2((float)(k * k)), add2(cs[3 + k], cs[3 - k]), e2);
    }
    return Q343PairSums{rho, jx, jy, jz, e2};
}

// rho, u, T of both nodes and their rotational values.
template <bool ROT, bool WHOLE, typename ST>
__device__ __forceinline__ void q343_pair_moments(const Params<kQ343, ST> &p, const PairOffsets &o, int rest,
                                                  const Q343PairSums &s, F2 (&h)[7], Moments &m0, Moments &m1)
{
    F2 R2 = f2(0.f);
    if (ROT) {
#pragma unroll
        for (int j = 0; j < 7; ++j) {
            const F2 w = f2(p.wr[j]);
            h[j] = fma2(w, Pair16<ST>::get(ld_pair<WHOLE>(p, kQ343 + j, rest, o, 0)), w);
        }
#pragma unroll
        for (int k = 1; k <= 3; ++k) R2 = fma2(f2((float)(k * k)), add2(h[3 + k], h[3 - k]), R2);
    }
    m0 = make_moments<3, ROT>(p, lo(s.rho), lo(s.jx), lo(s.jy), lo(s.jz), lo(s.e2), lo(R2));
    m1 = make_moments<3, ROT>(p, hi(s.rho), hi(s.jx), hi(s.jy), hi(s.jz), hi(s.e2), hi(R2));
}

// row_quartic of both nodes.
struct PairQuartic {
    F2 a00, a01, a02, a10, a11, a20, a21, k6, k24;  // EqCoef
    F2 v, v2, k3k6, k4k24, k6k24, a02x2, a21x2, b4;  // RowQuartic
};
__device__ __forceinline__ PairQuartic pair_quartic_setup(const EqCoef &k0, const EqCoef &k1, float v0, float v1,
                                                          float r2)
{
    const RowQuartic q0 = row_quartic_setup(k0, v0, r2), q1 = row_quartic_setup(k1, v1, r2);
    PairQuartic q;
    q.a00 = f2(k0.a00, k1.a00), q.a01 = f2(k0.a01, k1.a01), q.a02 = f2(k0.a02, k1.a02);
    q.a10 = f2(k0.a10, k1.a10), q.a11 = f2(k0.a11, k1.a11), q.a20 = f2(k0.a20, k1.a20);
    q.a21 = f2(k0.a21, k1.a21), q.k6 = f2(k0.k6, k1.k6), q.k24 = f2(k0.k24, k1.k24);
    q.v = f2(q0.v, q1.v), q.v2 = f2(q0.v2, q1.v2), q.k3k6 = f2(q0.k3k6, q1.k3k6);
    q.k4k24 = f2(q0.k4k24, q1.k4k24), q.k6k24 = f2(q0.k6k24, q1.k6k24);
    q.a02x2 = f2(q0.a02x2, q1.a02x2), q.a21x2 = f2(q0.a21x2, q1.a21x2), q.b4 = f2(q0.b4, q1.b4);
    return q;
}
__device__ __forceinline__ void pair_quartic(const PairQuartic &q, float r2f, F2 C0, float S0f, F2 (&P)[7])
{
    const F2 r2 = f2(r2f), S0 = f2(S0f);
    const F2 A0 = fma2(S0, fma2(S0, q.a02, q.a01), q.a00);
    const F2 A1 = fma2(S0, q.a11, q.a10);
    const F2 A2 = fma2(S0, q.a21, q.a20);
    const F2 b0 = fma2(C0, fma2(C0, fma2(C0, fma2(C0, q.k24, q.k6), A2), A1), A0);
    const F2 b1 = mul2(q.v, fma2(C0, fma2(C0, fma2(C0, q.k4k24, q.k3k6), add2(A2, A2)), A1));
    const F2 b2 = fma2(r2, fma2(C0, fma2(C0, q.a21, q.a11), fma2(q.a02x2, S0, q.a01)),
                       mul2(q.v2, fma2(C0, fma2(C0, q.k6k24, q.k3k6), A2)));
    const F2 b3 = mul2(q.v, fma2(r2, fma2(C0, q.a21x2, q.a11), mul2(q.v2, fma2(C0, q.k4k24, q.k6))));
    P[3] = b0;
#pragma unroll
    for (int m = 1; m <= 3; ++m) {
        const F2 E = fma2(q.b4, f2((float)(m * m * m * m)), fma2(b2, f2((float)(m * m)), b0));
        const F2 t = fma2(b3, f2((float)(m * m)), b1);  // the odd part is m t
        P[3 + m] = m == 1 ? add2(E, t) : fma2(f2((float)m), t, E);
        P[3 - m] = m == 1 ? sub2(E, t) : fma2(f2(-(float)m), t, E);
    }
}

// q343_collide of both nodes, on deviations.
template <bool ROT, int NS, int BLOCK, bool WHOLE, typename ST>
__device__ __forceinline__ void q343_pair_collide(const Params<kQ343, ST> &p, const Q343Weights &qw,
                                                  const PairOffsets &o, int x, int z, const Q343PairSums &s,
                                                  const uint32_t *stash)
{
    using V = Pair16<ST>;
    constexpr int C = (kQ343 - 1) / 2;
    const int plane = p.pitch * p.Y, rest = z * plane + o.y[3];
    F2 h[7];
    Moments m0, m1;
    q343_pair_moments<ROT, WHOLE>(p, o, rest, s, h, m0, m1);
    auto bad = [](const Moments &m) { return !(m.rho > 0.f) || !(m.T > 0.f) || !(fabsf(m.T) < 3.0e38f); };
    if (bad(m0) || (x + 1 < p.X && bad(m1))) atomicOr(p.status, 1);

    const float or0 = p.omega * m0.rho, or1 = p.omega * m1.rho;
    const EqCoef k0 = eq_coef<3>(m0.T, m0.ux * m0.ux + m0.uy * m0.uy + m0.uz * m0.uz, or0);
    const EqCoef k1 = eq_coef<3>(m1.T, m1.ux * m1.ux + m1.uy * m1.uy + m1.uz * m1.uz, or1);
    const PairQuartic q = pair_quartic_setup(k0, k1, m0.ux * p.r, m1.ux * p.r, p.r2);
    const F2 ruy = f2(m0.uy * p.r, m1.uy * p.r), ruz = f2(m0.uz * p.r, m1.uz * p.r);
    const F2 keep = f2(1.0f - p.omega), om = f2(p.omega);
    unsigned short *out = reinterpret_cast<unsigned short *>(p.dst) + (uint32_t)(rest + x);
    auto put = [&](int i, F2 d) { *reinterpret_cast<uint32_t *>(out + (uint64_t)i * (uint64_t)p.S) = V::put(d); };
    F2 acc0 = f2(0.f), acc2 = f2(0.f), ax = f2(0.f), ay = f2(0.f), az = f2(0.f);
    // P and the raw pair of the rest and the unit velocities, stored last
    F2 P_c, P_mx, P_px, P_my, P_py, P_mz, P_pz;
    uint32_t d_c = 0, d_mx = 0, d_px = 0, d_my = 0, d_py = 0, d_mz = 0, d_pz = 0;
    P_c = P_mx = P_px = P_my = P_py = P_mz = P_pz = f2(0.f);
    auto plane2 = [&](auto kept, int c) {
        constexpr bool KEPT = decltype(kept)::value;
        const int zo = bc_wrap(z - (c - 3), p.Z, p.bc2) * plane;
        const int ez = c - 3;
        const float ez2 = (float)(ez * ez);
        F2 p0 = f2(0.f), p2 = f2(0.f), px = f2(0.f), py = f2(0.f);
#pragma unroll
        for (int b = 0; b < 7; ++b) {
            const int row = zo + o.y[6 - b];
            const int ey = b - 3;
            const F2 cyz = fma2(f2((float)ey), ruy, mul2(f2((float)ez), ruz));
            const float eyz2 = (float)(ey * ey) + ez2;
            F2 Prow[7];
            pair_quartic(q, p.r2, cyz, p.r2 * eyz2, Prow);
            F2 r0 = f2(0.f), r2 = f2(0.f), rx = f2(0.f);
#pragma unroll
            for (int a = 0; a < 7; ++a) {
                const int ex = a - 3;
                const int i = (c * 7 + b) * 7 + a;
                const F2 P = Prow[a];
                r0 = fma2(f2(qw.w2[b * 7 + a]), P, r0);
                if (ex) {
                    r2 = fma2(f2(qw.w2x2[b * 7 + a]), P, r2);
                    rx = fma2(f2(qw.w2x[b * 7 + a]), P, rx);
                }
                uint32_t d;
                if constexpr (KEPT) d = stash[i * BLOCK + threadIdx.x];
                else d = ld_pair<WHOLE>(p, i, row, o, 3 - a);
                if (ex * ex + ey * ey <= 1 && ex * ex + ey * ey + ez * ez <= 1) {
                    if (ex == 0 && ey == 0 && ez == 0) { P_c = P; d_c = d; }
                    else if (ex == -1) { P_mx = P; d_mx = d; }
                    else if (ex == 1) { P_px = P; d_px = d; }
                    else if (ey == -1) { P_my = P; d_my = d; }
                    else if (ey == 1) { P_py = P; d_py = d; }
                    else if (ez == -1) { P_mz = P; d_mz = d; }
                    else { P_pz = P; d_pz = d; }
                } else {
                    put(i, fma2(keep, V::get(d), sub2(P, om)));
                }
            }
            p0 = add2(p0, r0);
            p2 = add2(p2, fma2(f2(eyz2), r0, r2));
            px = add2(px, rx);
            py = fma2(f2((float)ey), r0, py);
        }
        const F2 wc = f2(qw.wc[c]);
        acc0 = fma2(wc, p0, acc0);
        acc2 = fma2(wc, p2, acc2);
        ax = fma2(wc, px, ax);
        ay = fma2(wc, py, ay);
        az = fma2(f2(qw.wc[c] * (float)ez), p0, az);
    };
#pragma unroll 1
    for (int c = 6; c >= 0; --c) {
        if (c < NS) plane2(std::true_type{}, c);
        else plane2(std::false_type{}, c);
    }
    const F2 d0 = sub2(f2(or0, or1), acc0);
    const F2 d2 = fma2(om, f2(m0.E2_eq, m1.E2_eq), neg2(acc2));
    const F2 bb = mul2(d2, f2(0.5f / 3.0f));
    const F2 half = f2(0.5f);
    const F2 dmx = mul2(half, fma2(om, f2(m0.j[0], m1.j[0]), neg2(ax)));
    const F2 dmy = mul2(half, fma2(om, f2(m0.j[1], m1.j[1]), neg2(ay)));
    const F2 dmz = mul2(half, fma2(om, f2(m0.j[2], m1.j[2]), neg2(az)));
    const F2 iw0 = f2(qw.iw_rest), iw1 = f2(qw.iw_unit);
    auto last = [&](int i, uint32_t d, F2 P, F2 corr, F2 iw) {
        put(i, fma2(keep, V::get(d), fma2(corr, iw, sub2(P, om))));
    };
    last(C, d_c, P_c, sub2(d0, d2), iw0);
    last(C - 1, d_mx, P_mx, sub2(bb, dmx), iw1);
    last(C + 1, d_px, P_px, add2(bb, dmx), iw1);
    last(C - 7, d_my, P_my, sub2(bb, dmy), iw1);
    last(C + 7, d_py, P_py, add2(bb, dmy), iw1);
    last(C - 49, d_mz, P_mz, sub2(bb, dmz), iw1);
    last(C + 49, d_pz, P_pz, add2(bb, dmz), iw1);

    if (ROT) {
        // rows and planes: two upwind and one downwind of each node
        int rz[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) rz[k] = bc_wrap(z + k - 2, p.Z, p.bc2) * plane + o.y[3];
        auto load = [&](int j, int row) { return ld_pair<WHOLE>(p, kQ343 + j, row, o, 0); };
        pair_rot_update<ST>(
            p, m0, m1, h, [&](int j, int d) { return ld_pair<WHOLE>(p, kQ343 + j, rest, o, d); },
            [&](int j, int a, int d) { return load(j, a == 1 ? z * plane + o.y[3 + d] : rz[2 + d]); },
            [&](int j, F2 f) { put(kQ343 + j, fma2(f, f2(p.iwr[j]), f2(-1.0f))); });
    }
}

template <bool ROT, int BLOCK, bool WHOLE, typename ST>
__global__ void __launch_bounds__(BLOCK, kPairWarps * 32 / BLOCK)
    k_step_q343_pair(const Params<kQ343, ST> p, const Q343Weights qw)
{
    const int x = 2 * (blockIdx.x * BLOCK + threadIdx.x);
    const int y = blockIdx.y, z = blockIdx.z;
    if (x >= p.X) return;
    const PairOffsets o = pair_offsets(p, x, y);
    extern __shared__ unsigned char q343_smem[];
    uint32_t *stash = reinterpret_cast<uint32_t *>(q343_smem);
    const Q343PairSums s = q343_pair_sums<kPairStash, BLOCK, WHOLE>(p, o, z, stash);
    q343_pair_collide<ROT, kPairStash, BLOCK, WHOLE>(p, qw, o, x, z, s, stash);
}

// The sums for the moments alone, opposite velocities before the rest
// (q343_moment_sums below) of both nodes.
template <bool WHOLE, typename ST>
__device__ __forceinline__ Q343PairSums q343_pair_moment_sums(const Params<kQ343, ST> &p, const PairOffsets &o, int z)
{
    const int plane = p.pitch * p.Y;
    F2 cs[7], rs[7];
#pragma unroll
    for (int a = 0; a < 7; ++a) cs[a] = rs[a] = f2(0.f);
    auto add = [&](int c) {  // the sum of the plane of e_z = c - 3
        const int zo = bc_wrap(z - (c - 3), p.Z, p.bc2) * plane;
        F2 sum = f2(0.f);
#pragma unroll
        for (int b = 0; b < 7; ++b) {
            const int row = zo + o.y[6 - b];
            F2 rsum = f2(0.f);
#pragma unroll
            for (int a = 0; a < 7; ++a) {
                const int i = (c * 7 + b) * 7 + a;
                const F2 w = f2(p.w[i]);
                const F2 g = fma2(w, Pair16<ST>::get(ld_pair<WHOLE>(p, i, row, o, 3 - a)), w);
                cs[a] = add2(cs[a], g);
                rsum = a ? add2(rsum, g) : g;
            }
            rs[b] = add2(rs[b], rsum);
            sum = add2(sum, rsum);
        }
        return sum;
    };
    Q343PairSums s{f2(0.f), f2(0.f), f2(0.f), f2(0.f), f2(0.f)};
#pragma unroll 1
    for (int k = 3; k >= 1; --k) {
        const F2 lo = add(3 - k), hi = add(3 + k);
        s.jz = fma2(f2((float)k), sub2(hi, lo), s.jz);
        s.e2 = fma2(f2((float)(k * k)), add2(hi, lo), s.e2);
    }
    add(3);
    s.rho = cs[3];
#pragma unroll
    for (int k = 1; k <= 3; ++k) {
        const F2 d = f2((float)k), dd = f2((float)(k * k)), sx = add2(cs[3 + k], cs[3 - k]);
        s.rho = add2(s.rho, sx);
        s.jx = fma2(d, sub2(cs[3 + k], cs[3 - k]), s.jx);
        s.jy = fma2(d, sub2(rs[3 + k], rs[3 - k]), s.jy);
        s.e2 = fma2(dd, sx, s.e2);
        s.e2 = fma2(dd, add2(rs[3 + k], rs[3 - k]), s.e2);
    }
    return s;
}

template <bool ROT, bool WHOLE, typename ST>
__global__ void __launch_bounds__(kQ343Block, 4) k_moments_q343_pair(const Params<kQ343, ST> p)
{
    const int x = 2 * (blockIdx.x * kQ343Block + threadIdx.x);
    const int y = blockIdx.y, z = blockIdx.z;
    if (x >= p.X) return;
    const PairOffsets o = pair_offsets(p, x, y);
    const Q343PairSums s = q343_pair_moment_sums<WHOLE>(p, o, z);
    F2 h[7];
    Moments m[2];
    q343_pair_moments<ROT, WHOLE>(p, o, z * p.pitch * p.Y + o.y[3], s, h, m[0], m[1]);
    const int64_t node = ((int64_t)z * p.Y + y) * p.X + x;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        if (x + k >= p.X) break;
        p.out0[node + k] = m[k].rho;
        p.out1[node + k] = m[k].ux;
        p.out1[p.N + node + k] = m[k].uy;
        p.out1[2 * p.N + node + k] = m[k].uz;
        p.out2[node + k] = m[k].T;
    }
}

// Float storage, one launch: pass 1, then pass 2 on the same thread.  The two
// step kernels are not launched dependently: pass 2 interleaves its loads with
// its stores and needs the read-only path (see ld), which a kernel that is
// resident while its predecessor writes may not use.  With ordinary loads and
// the dependent launch, the next row loaded ahead: 101 x 96 x 90 float n = 4
// 0.83-0.89 ms a step against 0.775; 256^3 half n = 0 / n = 4 8.15 / 9.13
// against 7.70 / 8.63.
template <bool ROT>
__global__ void __launch_bounds__(kQ343Block, LBM_Q343_MIN_BLOCKS)
    k_step_q343(const Params<kQ343> p, const Q343Weights qw)
{
    const int x = blockIdx.x * kQ343Block + threadIdx.x;
    const int y = blockIdx.y, z = blockIdx.z;
    if (x >= p.X) return;
    const Offsets o = node_offsets<3>(p, x, y, z);
    q343_collide<ROT>(p, qw, o, z, q343_sums(p, o, z));
}

// The five sums for the moments alone: by e_x, e_y and e_z first, opposite
// velocities before the rest, as node_moments takes them (no sum has more than 49
// terms in a row, and a mirror-symmetric state gives exactly zero momentum).
__device__ __forceinline__ Q343Sums q343_moment_sums(const Params<kQ343> &p, const Offsets &o, int z)
{
    const int plane = p.pitch * p.Y;
    float cs[7], rs[7];
#pragma unroll
    for (int a = 0; a < 7; ++a) cs[a] = rs[a] = 0.f;
    auto add = [&](int c) {  // the sum of the plane of e_z = c - 3
        const int zo = bc_wrap(z - (c - 3), p.Z, p.bc2) * plane;
        float sum = 0.f;
#pragma unroll
        for (int b = 0; b < 7; ++b) {
            const int row = zo + o.y[6 - b];
            float rsum = 0.f;
#pragma unroll
            for (int a = 0; a < 7; ++a) {
                const float g = q343_load(p, (c * 7 + b) * 7 + a, row + o.x[6 - a]);
                cs[a] += g;
                rsum += g;
            }
            rs[b] += rsum;
            sum += rsum;
        }
        return sum;
    };
    Q343Sums s{0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
    for (int k = 3; k >= 1; --k) {
        const float lo = add(3 - k), hi = add(3 + k), d = (float)k;
        s.jz = fmaf(d, hi - lo, s.jz);
        s.e2 = fmaf(d * d, hi + lo, s.e2);
    }
    add(3);
    s.rho = cs[3];
#pragma unroll
    for (int k = 1; k <= 3; ++k) {
        const float d = (float)k, sx = cs[3 + k] + cs[3 - k];
        s.rho += sx;
        s.jx = fmaf(d, cs[3 + k] - cs[3 - k], s.jx);
        s.jy = fmaf(d, rs[3 + k] - rs[3 - k], s.jy);
        s.e2 = fmaf(d * d, sx, s.e2);
        s.e2 = fmaf(d * d, rs[3 + k] + rs[3 - k], s.e2);
    }
    return s;
}

// rho, u, T of the current state: pass 1 of the step and the rotational
// energy, nothing kept (no stash, no per-node array of the 343 values: that
// array, in local memory, is what the general k_moments spent its time on).
// Bound by issue and load latency, as pass 1 of the step is: 101 x 96 x 90
// float n = 4 0.241 ms (0.860 with k_moments); 256^3 half, two nodes per
// thread below, 2.30 ms (3.12 with one, 14.6 with k_moments).
template <bool ROT> __global__ void __launch_bounds__(kQ343Block, 4) k_moments_q343(const Params<kQ343> p)
{
    const int x = blockIdx.x * kQ343Block + threadIdx.x;
    const int y = blockIdx.y, z = blockIdx.z;
    if (x >= p.X) return;
    const Offsets o = node_offsets<3>(p, x, y, z);
    const Q343Sums s = q343_moment_sums(p, o, z);
    float R2 = 0.f;
    if (ROT) {
#pragma unroll
        for (int k = 1; k <= 3; ++k)
            R2 = fmaf((float)(k * k), ld(p, kQ343 + 3 + k, o.self()) + ld(p, kQ343 + 3 - k, o.self()), R2);
    }
    const Moments m = make_moments<3, ROT>(p, s.rho, s.jx, s.jy, s.jz, s.e2, R2);
    const int64_t node = ((int64_t)z * p.Y + y) * p.X + x;
    p.out0[node] = m.rho;
    p.out1[node] = m.ux;
    p.out1[p.N + node] = m.uy;
    p.out1[2 * p.N + node] = m.uz;
    p.out2[node] = m.T;
}

}  // namespace

template <bool ROT, typename ST> cudaError_t launch_moments_q343(const Args &a, cudaStream_t s)
{
    const auto p = make_params<kQ343, ST>(a);
    if constexpr (!std::is_same<ST, float>::value) {
        const dim3 pairs((a.X + 2 * kQ343Block - 1) / (2 * kQ343Block), a.Y, a.Z);
        if (pair_whole(a)) k_moments_q343_pair<ROT, true><<<pairs, kQ343Block, 0, s>>>(p);
        else k_moments_q343_pair<ROT, false><<<pairs, kQ343Block, 0, s>>>(p);
        return cudaGetLastError();
    } else {
    const dim3 grid((a.X + kQ343Block - 1) / kQ343Block, a.Y, a.Z);
    k_moments_q343<ROT><<<grid, kQ343Block, 0, s>>>(p);
    return cudaGetLastError();
    }
}

template <bool ROT, typename ST> cudaError_t launch_step_q343(const Args &a, cudaStream_t s)
{
    const auto p = make_params<kQ343, ST>(a);
    Q343Weights qw;
    for (int b = 0; b < 7; ++b)
        for (int c = 0; c < 7; ++c) {
            const double wab = (double)a.wr[c] * (double)a.wr[b];
            qw.w2[b * 7 + c] = (float)wab;
            qw.w2x[b * 7 + c] = (float)(wab * (c - 3));
            qw.w2x2[b * 7 + c] = (float)(wab * (c - 3) * (c - 3));
        }
    for (int c = 0; c < 7; ++c) qw.wc[c] = a.wr[c];
    qw.iw_rest = (float)(1.0 / ((double)a.wr[3] * (double)a.wr[3] * (double)a.wr[3]));
    qw.iw_unit = (float)(1.0 / ((double)a.wr[2] * (double)a.wr[3] * (double)a.wr[3]));
    if constexpr (std::is_same<ST, float>::value) {
        const dim3 grid((a.X + kQ343Block - 1) / kQ343Block, a.Y, a.Z);
        k_step_q343<ROT><<<grid, kQ343Block, 0, s>>>(p, qw);
        return cudaGetLastError();
    } else {
        auto go = [&](auto whole, auto block) {
            constexpr bool W = decltype(whole)::value;
            constexpr int B = decltype(block)::value;
            constexpr size_t smem = pair_stash_bytes<B>();
            const cudaError_t e = allow_smem<k_step_q343_pair<ROT, B, W, ST>>(smem);
            if (e != cudaSuccess) return e;
            const dim3 grid((a.X + 2 * B - 1) / (2 * B), a.Y, a.Z);
            k_step_q343_pair<ROT, B, W, ST><<<grid, B, smem, s>>>(p, qw);
            return cudaGetLastError();
        };
        const bool odd = (a.X + 63) / 64 % 2;
        using B32 = std::integral_constant<int, 32>;
        using B64 = std::integral_constant<int, 64>;
        if (pair_whole(a)) return odd ? go(std::true_type{}, B32{}) : go(std::true_type{}, B64{});
        return odd ? go(std::false_type{}, B32{}) : go(std::false_type{}, B64{});
    }
}

cudaError_t launch_d3q343(Op op, const Args &a, cudaStream_t s) { return launch_lattice<4>(op, a, s); }

}  // namespace lbm
