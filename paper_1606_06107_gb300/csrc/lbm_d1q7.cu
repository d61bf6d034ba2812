// Kernel instantiations for the D1Q7 lattice, and its float steps: one launch
// per step, or many steps of one tube in one launch (lbm_tube.cuh has the
// node update).
#include <algorithm>
#include <cooperative_groups.h>

#include "lbm_tube.cuh"

namespace lbm {
namespace {

namespace cg = cooperative_groups;

struct TubeParams {
    TubeLattice lat;
    TubeRates rates;
    const float *src;
    float *dst;
    int *status;
    int64_t S;
    int X, bc;
};

TubeParams tube_params(const Args &a)
{
    TubeParams p{};
    p.lat = tube_lattice(a.w, a.r, a.nu_scale, a.inv_m);
    p.rates = tube_rates(a.omega, a.cT, a.half_n);
    p.src = static_cast<const float *>(a.src);
    p.dst = static_cast<float *>(a.dst);
    p.status = a.status;
    p.S = a.S;
    p.X = a.X;
    p.bc = a.bc[0];
    return p;
}

// One step, one node per thread.
template <bool ROT, int MODE> __global__ void __launch_bounds__(kBlockX) k_tube_step(const TubeParams p)
{
    const int x = blockIdx.x * kBlockX + threadIdx.x;
    if (x >= p.X) return;
    int o[7];
#pragma unroll
    for (int k = 0; k < 7; ++k) o[k] = bc_wrap(x + k - 3, p.X, p.bc);
    pdl_wait();
    pdl_trigger();
    float out[ROT ? 14 : 7], rho, T;
    tube_update<ROT, MODE>(
        p.lat, p.rates, [&](int pop, int d) { return __ldca(p.src + ((uint32_t)pop * (uint32_t)p.S + (uint32_t)o[3 + d])); },
        [&](float ux) {
            const bool pos = ux >= 0.f;
            const int u2 = pos ? o[1] : o[5], u1 = pos ? o[2] : o[4], d1 = pos ? o[4] : o[2];
            return [&p, u2, u1, d1](int j, int k) {
                return __ldca(p.src + ((uint32_t)(7 + j) * (uint32_t)p.S + (uint32_t)(k == 2 ? u2 : k == 1 ? u1 : d1)));
            };
        },
        out, rho, T);
#pragma unroll
    for (int i = 0; i < (ROT ? 14 : 7); ++i) p.dst[(uint32_t)i * (uint32_t)p.S + (uint32_t)x] = out[i];
    if (tube_bad(rho, T)) atomicOr(p.status, 1);
}

// `steps` steps of one tube by one cluster.  A tube of a few thousand nodes is
// a handful of blocks, so one launch per step costs the launch (4.1 us on a
// 1000-node tube), not the work.  Here up to eight blocks each keep a piece of
// the tube in shared memory, two copies of the state and a halo of three nodes
// on each side; a step computes the piece from one copy into the other, stores
// the piece's outer nodes into the neighbours' halos as well (distributed
// shared memory), and ends in one cluster barrier.  The state lies node by
// node, 15 floats apart (14 populations; odd, so that consecutive lanes take
// different banks): every population and neighbour is an immediate offset from
// one address.  A copy end keeps three copies of its node in the halo.
// Bound by the latency of one node update and the barrier: 1000 nodes, FD, n =
// 4, 0.75 us per step (4.1 with a launch each).
constexpr int kTubeCluster = 8;      // blocks per cluster (the portable limit)
constexpr int kTubeMinPiece = 32;    // nodes a block owns at least: a warp
constexpr int kTubeMaxPiece = 1024;  // and at most: a node a thread
constexpr int kNodePitch = 15;

// MAXT: most threads a block.  Pieces of up to 256 nodes (tubes of 2048) may
// use the registers that 1024 threads cannot have.
template <bool ROT, int MODE, int MAXT>
__global__ void __launch_bounds__(MAXT) k_tube_steps(const TubeParams p, int64_t steps, int nodes)
{
    extern __shared__ float tube_smem[];  // [2][nodes][kNodePitch]
    constexpr int POPS = ROT ? 14 : 7;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), blocks = (int)cluster.num_blocks();
    auto first = [&](int r) { return (int)((int64_t)p.X * r / blocks); };
    const int c0 = first(rank), n = first(rank + 1) - c0;
    const bool wrap = p.bc == 0;
    const int left = rank ? rank - 1 : blocks - 1, right = rank + 1 < blocks ? rank + 1 : 0;
    const bool has_left = wrap || rank > 0, has_right = wrap || rank + 1 < blocks;
    const int n_left = first(left + 1) - first(left);
    float *a = tube_smem, *b = tube_smem + nodes * kNodePitch;
    // local node l + 3 is node c0 + l
    for (int l = threadIdx.x; l < n + 6; l += blockDim.x) {
        const int x = bc_wrap(c0 + l - 3, p.X, p.bc);
#pragma unroll
        for (int i = 0; i < POPS; ++i) a[l * kNodePitch + i] = __ldcg(p.src + (size_t)i * p.S + x);
    }
    cluster.sync();  // every block has started: its shared memory can be written
    const int l = threadIdx.x;
    for (int64_t s = 0; s < steps; ++s) {
        if (l < n) {
            const float *me = a + (l + 3) * kNodePitch;
            float out[POPS], rho, T;
            tube_update<ROT, MODE>(
                p.lat, p.rates, [&](int pop, int d) { return me[d * kNodePitch + pop]; },
                [&](float ux) {
                    const int up = ux >= 0.f ? -kNodePitch : kNodePitch;
                    const float *u1 = me + up, *u2 = me + 2 * up, *d1 = me - up;
                    return [u1, u2, d1](int j, int k) { return (k == 2 ? u2 : k == 1 ? u1 : d1)[7 + j]; };
                },
                out, rho, T);
            if (tube_bad(rho, T)) atomicOr(p.status, 1);
            auto put = [&](float *base, int at) {
#pragma unroll
                for (int i = 0; i < POPS; ++i) base[at * kNodePitch + i] = out[i];
            };
            put(b, l + 3);
            if (has_left && l < 3) put(cluster.map_shared_rank(b, left), n_left + 3 + l);
            if (has_right && l >= n - 3) put(cluster.map_shared_rank(b, right), l - (n - 3));
            if (!has_left && l == 0)
                for (int k = 0; k < 3; ++k) put(b, k);
            if (!has_right && l == n - 1)
                for (int k = 0; k < 3; ++k) put(b, n + 3 + k);
        }
        float *t = a;
        a = b;
        b = t;
        cluster.sync();  // step s + 1 reads what the neighbours wrote, and may overwrite what they read
    }
    if (l < n) {
#pragma unroll
        for (int i = 0; i < POPS; ++i) p.dst[(size_t)i * p.S + c0 + l] = a[(l + 3) * kNodePitch + i];
    }
}

template <bool ROT, int MODE, int MAXT> cudaError_t launch_tube_t(const Args &a, int64_t steps, cudaStream_t s)
{
    const TubeParams p = tube_params(a);
    // as many blocks as leave each at least a warp of nodes
    const int blocks = std::min(kTubeCluster, std::max(1, a.X / kTubeMinPiece));
    const int piece = (a.X + blocks - 1) / blocks, nodes = piece + 6;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3((piece + 31) / 32 * 32);
    cfg.dynamicSmemBytes = sizeof(float) * 2 * kNodePitch * nodes;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = blocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = allow_smem<k_tube_steps<ROT, MODE, MAXT>>(sizeof(float) * 2 * kNodePitch * (MAXT + 6));
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, k_tube_steps<ROT, MODE, MAXT>, p, steps, nodes);
}

template <bool ROT, int MODE> cudaError_t launch_tube(const Args &a, int64_t steps, cudaStream_t s)
{
    if (steps == 1) {
        const dim3 grid((a.X + kBlockX - 1) / kBlockX);
        return launch_pdl(k_tube_step<ROT, MODE>, grid, dim3(kBlockX), 0, s, tube_params(a));
    }
    return a.X <= kTubeCluster * 256 ? launch_tube_t<ROT, MODE, 256>(a, steps, s)
                                     : launch_tube_t<ROT, MODE, kTubeMaxPiece>(a, steps, s);
}

}  // namespace

// Whether `steps` steps of this problem run as one launch: float storage, a
// tube whose pieces fit one node a thread (8192 nodes, where a block of 1024
// threads still takes less than the launch and eight times the blocks gain
// little), long enough for a halo beside every piece, and enough steps to pay
// for loading and storing the state.
bool tube_steps_ok(const Args &a, int64_t steps)
{
    return a.storage == 0 && a.X >= kTubeMinPiece && a.X <= kTubeCluster * kTubeMaxPiece && steps >= 4;
}

cudaError_t launch_tube_steps(const Args &a, int64_t steps, cudaStream_t s)
{
    if (a.Qr > 0) return a.mode ? launch_tube<true, 1>(a, steps, s) : launch_tube<true, 0>(a, steps, s);
    return a.mode ? launch_tube<false, 1>(a, steps, s) : launch_tube<false, 0>(a, steps, s);
}

cudaError_t launch_d1q7(Op op, const Args &a, cudaStream_t s)
{
    if (op == Op::Step && a.storage == 0) return launch_tube_steps(a, 1, s);
    return launch_lattice<1>(op, a, s);
}
}  // namespace lbm
