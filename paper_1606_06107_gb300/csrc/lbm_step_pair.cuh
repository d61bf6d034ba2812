// Two x-adjacent nodes per thread for half and bfloat16 deviations from rest:
// the pieces that the D3Q343 step (lbm_d3q343.cu) and the 2-D moments below
// share.  Included by lbm_step.cuh inside namespace lbm.
//
// With 16-bit values a node moves half of float's bytes and one node per
// thread is bound by instruction issue, a third of it address arithmetic,
// conversions and 2-byte memory operations at half rate.  Here a thread owns
// nodes x and x + 1, x even: every floating-point operation is a packed one on
// both (f32x2: the pipe takes as long, the issue slot is shared), a population
// that moves an even number of nodes is one aligned 32-bit load for both, an
// odd one two 16-bit loads, and every store is 32 bits.
//
// The 2-D step in this form was measured and dropped: 300 us on the 2048^2
// D2Q49 half state against 313 for k_step (2888 instructions per pair, 128
// registers, load latency), and the contraction of its multiply-adds differs
// from k_step's, which 16-bit rounding shows at 3e-5 of u after ten steps.
#pragma once

// ---- two floats in one register pair --------------------------------------
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 f2(float lo, float hi)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ F2 f2(float s) { return f2(s, s); }
__device__ __forceinline__ float lo(F2 a)
{
    float l, h;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(l), "=f"(h) : "l"(a.v));
    return l;
}
__device__ __forceinline__ float hi(F2 a)
{
    float l, h;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(l), "=f"(h) : "l"(a.v));
    return h;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b)
{
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 add2(F2 a, F2 b)
{
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 sub2(F2 a, F2 b)
{
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}

__device__ __forceinline__ F2 neg2(F2 a) { return F2{a.v ^ 0x8000000080000000ull}; }

// ---- two 16-bit values in one register -------------------------------------
template <typename ST> struct Pair16;
template <> struct Pair16<__half> {
    __device__ __forceinline__ static F2 get(uint32_t q)
    {
        const __half2 h = *reinterpret_cast<const __half2 *>(&q);
        return f2(__low2float(h), __high2float(h));
    }
    __device__ __forceinline__ static uint32_t put(F2 v)
    {
        const __half2 h = __floats2half2_rn(lo(v), hi(v));
        return *reinterpret_cast<const uint32_t *>(&h);
    }
};
template <> struct Pair16<__nv_bfloat16> {
    __device__ __forceinline__ static F2 get(uint32_t q)
    {
        return f2(__uint_as_float(q << 16), __uint_as_float(q & 0xffff0000u));
    }
    __device__ __forceinline__ static uint32_t put(F2 v)
    {
        const __nv_bfloat162 h = __floats2bfloat162_rn(lo(v), hi(v));
        return *reinterpret_cast<const uint32_t *>(&h);
    }
};

// Element offsets x - 3 .. x + 4 and rows y - 3 .. y + 3 of a thread's pair.
// (Column x + 4 only serves node x + 1; where that is past an odd row's end
// the offset may be the row's first padding element, which is in the buffer.)
struct PairOffsets {
    int x[8], y[7];
};
template <int Q, typename ST>
__device__ __forceinline__ PairOffsets pair_offsets(const Params<Q, ST> &p, int x, int y)
{
    PairOffsets o;
#pragma unroll
    for (int k = 0; k < 8; ++k) o.x[k] = bc_wrap(x + k - 3, p.X, p.bc0);
#pragma unroll
    for (int k = 0; k < 7; ++k) o.y[k] = bc_wrap(y + k - 3, p.Y, p.bc1) * p.pitch;
    return o;
}

// The raw values of population `pop` at columns x + d and x + d + 1 of the row
// at offset `row`.  WHOLE: the pairs of even d are aligned words that the
// boundary never splits (a periodic axis of even extent).
// (Addresses formed from a 32- or 64-bit element index: with the population's
// base in uniform registers and a 32-bit byte offset per thread the 256^3
// D3Q343 step took 8.55 ms against 7.39.)
template <bool WHOLE, int Q, typename ST>
__device__ __forceinline__ uint32_t ld_pair(const Params<Q, ST> &p, int pop, int row, const PairOffsets &o, int d)
{
    using Idx = typename std::conditional<(Q > 49), uint64_t, uint32_t>::type;
    const unsigned short *src = reinterpret_cast<const unsigned short *>(p.src);
    const Idx at = (Idx)pop * (Idx)p.S + (Idx)(uint32_t)row;
    if (WHOLE && (d & 1) == 0)
        return ld_ro(reinterpret_cast<const uint32_t *>(src + (at + (Idx)(uint32_t)o.x[d + 3])));
    const uint32_t a = ld_ro(src + (at + (Idx)(uint32_t)o.x[d + 3]));
    const uint32_t b = ld_ro(src + (at + (Idx)(uint32_t)o.x[d + 4]));
    return __byte_perm(a, b, 0x5410);
}

// Pull of both nodes: the raw pairs.
template <int LAT, bool ROT, bool WHOLE, typename ST>
__device__ __forceinline__ void pair_pull(const Params<Lattice<LAT>::Q, ST> &p, const PairOffsets &o, uint32_t *graw,
                                          uint32_t *hraw)
{
    using L = Lattice<LAT>;
    static_for<0, L::Q>([&](auto ic) {
        constexpr int I = decltype(ic)::value;
        graw[I] = ld_pair<WHOLE>(p, I, o.y[3 - L::ey(I)], o, -L::ex(I));
    });
    if (ROT) {
#pragma unroll
        for (int j = 0; j < 7; ++j)
            hraw[j] = ld_pair<WHOLE>(p, L::Q + j, o.y[3], o, 0);
    }
}

// node_moments of both nodes.
template <int LAT, bool ROT, typename ST>
__device__ __forceinline__ void pair_moments(const Params<Lattice<LAT>::Q, ST> &p, const uint32_t *graw,
                                             const F2 *h, Moments &m0, Moments &m1)
{
    using L = Lattice<LAT>;
    F2 cs[7], rs[7];
    bool hc[7] = {}, hr[7] = {};
    static_for<0, L::Q>([&](auto ic) {
        constexpr int I = decltype(ic)::value;
        constexpr int a = L::ex(I) + 3, b = L::ey(I) + 3;
        const F2 w = f2(p.w[I]);
        const F2 g = fma2(w, Pair16<ST>::get(graw[I]), w);
        cs[a] = hc[a] ? add2(cs[a], g) : g;
        rs[b] = hr[b] ? add2(rs[b], g) : g;
        hc[a] = hr[b] = true;
    });
    F2 rho = cs[3], jx = f2(0.f), jy = f2(0.f), e2 = f2(0.f);
#pragma unroll
    for (int k = 1; k <= 3; ++k) {
        const F2 d = f2((float)k), dd = f2((float)(k * k));
        const F2 sx = add2(cs[3 + k], cs[3 - k]);
        rho = add2(rho, sx);
        jx = fma2(d, sub2(cs[3 + k], cs[3 - k]), jx);
        e2 = fma2(dd, sx, e2);
        jy = fma2(d, sub2(rs[3 + k], rs[3 - k]), jy);
        e2 = fma2(dd, add2(rs[3 + k], rs[3 - k]), e2);
    }
    F2 R2 = f2(0.f);
    if (ROT) {
#pragma unroll
        for (int k = 1; k <= 3; ++k) R2 = fma2(f2((float)(k * k)), add2(h[3 + k], h[3 - k]), R2);
    }
    m0 = make_moments<2, ROT>(p, lo(rho), lo(jx), lo(jy), 0.f, lo(e2), lo(R2));
    m1 = make_moments<2, ROT>(p, hi(rho), hi(jx), hi(jy), 0.f, hi(e2), hi(R2));
}

// rot_advect and rot_store of both nodes in three dimensions.  along(j, d): the raw pair of h_j at
// columns x + d, x + d + 1 of the nodes' own row; across(j, axis, d): the pair
// of the row (axis 1) or plane (axis 2) d nodes further; put(j, f) stores.
// The columns x - 2 .. x + 3 and four rows serve both signs of both nodes'
// velocities, so nothing is loaded twice and no lane waits for another's sign.
template <typename ST, int Q, typename Along, typename Across, typename Put>
__device__ __forceinline__ void pair_rot_update(const Params<Q, ST> &p, const Moments &m0, const Moments &m1,
                                                const F2 *h, Along &&along, Across &&across, Put &&put)
{
    using V = Pair16<ST>;
    const float n0[3] = {m0.ux * p.nu_scale, m0.uy * p.nu_scale, m0.uz * p.nu_scale};
    const float n1[3] = {m1.ux * p.nu_scale, m1.uy * p.nu_scale, m1.uz * p.nu_scale};
    const F2 keep = f2(1.0f - p.omega), om = f2(p.omega);
    float q0[7], q1[7];
    heq_node(p, m0.T, m0.T_lat, q0);
    heq_node(p, m1.T, m1.T_lat, q1);
    auto upwind = [](F2 a, F2 fuu, F2 fu, F2 f0, F2 fd, F2 adv) {
        F2 t = fma2(f2(-6.0f), fu, fuu);
        t = fma2(f2(3.0f), f0, t);
        t = fma2(f2(2.0f), fd, t);
        return fma2(a, mul2(t, f2(1.0f / 6.0f)), adv);
    };
#pragma unroll
    for (int j = 0; j < 7; ++j) {
        const F2 w = f2(p.wr[j]);
        auto decode = [&](uint32_t v) { return fma2(w, V::get(v), w); };
        F2 adv = f2(0.f);
        {
            const bool p0 = n0[0] >= 0.f, p1 = n1[0] >= 0.f;
            const F2 l = decode(along(j, -2)), r = decode(along(j, 2));
            adv = upwind(f2(fabsf(n0[0]), fabsf(n1[0])), f2(p0 ? lo(l) : lo(r), p1 ? hi(l) : hi(r)),
                         f2(p0 ? hi(l) : hi(h[j]), p1 ? lo(h[j]) : lo(r)), h[j],
                         f2(p0 ? hi(h[j]) : hi(l), p1 ? lo(r) : lo(h[j])), adv);
        }
#pragma unroll
        for (int a = 1; a < 3; ++a) {
            const bool p0 = n0[a] >= 0.f, p1 = n1[a] >= 0.f;
            const F2 b2 = decode(across(j, a, -2)), b1 = decode(across(j, a, -1));
            const F2 t1 = decode(across(j, a, 1)), t2 = decode(across(j, a, 2));
            adv = upwind(f2(fabsf(n0[a]), fabsf(n1[a])), f2(p0 ? lo(b2) : lo(t2), p1 ? hi(b2) : hi(t2)),
                         f2(p0 ? lo(b1) : lo(t1), p1 ? hi(b1) : hi(t1)), h[j],
                         f2(p0 ? lo(t1) : lo(b1), p1 ? hi(t1) : hi(b1)), adv);
        }
        put(j, fma2(keep, h[j], fma2(om, f2(q0[j], q1[j]), neg2(adv))));
    }
}

// rho, u, T on the 2-D lattices, STREAM transport: 137 us on the 2048^2 D2Q49
// half state (157 with one node per thread).
template <int LAT, bool ROT, bool WHOLE, typename ST>
__global__ void __launch_bounds__(kBlockX) k_moments_pair(const Params<Lattice<LAT>::Q, ST> p)
{
    using V = Pair16<ST>;
    const int x = 2 * (blockIdx.x * kBlockX + threadIdx.x), y = blockIdx.y;
    if (x >= p.X) return;
    const PairOffsets o = pair_offsets(p, x, y);
    uint32_t graw[Lattice<LAT>::Q], hraw[7];
    pair_pull<LAT, ROT, WHOLE>(p, o, graw, hraw);
    F2 h[7];
    if (ROT) {
#pragma unroll
        for (int j = 0; j < 7; ++j) {
            const F2 w = f2(p.wr[j]);
            h[j] = fma2(w, V::get(hraw[j]), w);
        }
    }
    Moments m[2];
    pair_moments<LAT, ROT>(p, graw, h, m[0], m[1]);
    const int64_t node = (int64_t)y * p.X + x;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        if (x + q >= p.X) break;
        p.out0[node + q] = m[q].rho;
        p.out1[node + q] = m[q].ux;
        p.out1[p.N + node + q] = m[q].uy;
        p.out2[node + q] = m[q].T;
    }
}
