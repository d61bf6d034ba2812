// Kernel instantiations for the D1Q7 lattice, and its many-step kernel for
// single tubes.
#include <algorithm>
#include <cooperative_groups.h>

#include "lbm_step.cuh"

namespace lbm {
namespace {

namespace cg = cooperative_groups;

// `steps` steps of one tube by one cluster.  A tube of a few thousand nodes is
// a handful of blocks, so one launch per step costs the launch (4.1 us on a
// 1000-node tube), not the work.  Here up to eight blocks each keep a piece of
// the tube in shared memory, two copies of the state and a halo of three nodes
// on each side; a step computes the piece from one copy into the other, stores
// the piece's outer nodes into the neighbours' halos as well (distributed
// shared memory), and ends in one cluster barrier.  The node update is
// k_step's (this file is compiled without multiply-add contraction), so the
// results are the same bits.  Bound by the latency of one node update and the
// barrier: 1000 nodes, FD, n = 4, 1.0 us per step (4.1 with a launch each).
constexpr int kTubeCluster = 8;     // blocks per cluster (the portable limit)
constexpr int kTubeMinPiece = 32;   // nodes a block owns at least: a warp
constexpr int kTubeMaxPiece = 1024; // and at most: a node a thread

// MAXT: most threads a block.  Pieces of up to 256 nodes (tubes of 2048) may
// use the registers that 1024 threads cannot have (28-40 bytes of spill there).
template <bool ROT, int MODE, int MAXT>
__global__ void __launch_bounds__(MAXT) k_tube_steps(const Params<7> p, int64_t steps, int pitch)
{
    extern __shared__ float tube_smem[];
    constexpr int POPS = ROT ? 14 : 7;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), blocks = (int)cluster.num_blocks();
    auto first = [&](int r) { return (int)((int64_t)p.X * r / blocks); };
    const int c0 = first(rank), n = first(rank + 1) - c0;
    const bool wrap = p.bc0 == 0;
    const int left = rank ? rank - 1 : blocks - 1, right = rank + 1 < blocks ? rank + 1 : 0;
    const bool has_left = wrap || rank > 0, has_right = wrap || rank + 1 < blocks;
    const int n_left = first(left + 1) - first(left);
    float *a = tube_smem, *b = tube_smem + POPS * pitch;
    // local index l + 3 is node c0 + l
    for (int l = threadIdx.x; l < n + 6; l += blockDim.x) {
        const int x = bc_wrap(c0 + l - 3, p.X, p.bc0);
#pragma unroll
        for (int i = 0; i < POPS; ++i) a[i * pitch + l] = __ldcg(p.src + (size_t)i * p.S + x);
    }
    cluster.sync();  // every block has started: its shared memory can be written
    const int l = threadIdx.x;
    Offsets o;
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        const int x = c0 + l + k - 3;
        o.x[k] = (wrap ? x : min(max(x, 0), p.X - 1)) - c0 + 3;
        o.y[k] = o.z[k] = 0;
    }
    for (int64_t s = 0; s < steps; ++s) {
        if (l < n) {
            Params<7> q = p;
            q.src = a;
            q.dst = b;
            q.S = pitch;
            float g[7], h[7];
            load_node<1, ROT, MODE, 2>(q, o, g, h);
            const Moments m = node_moments<1, ROT>(q, g, h);
            if (!(m.rho > 0.f) || !(m.T > 0.f) || !(fabsf(m.T) < 3.0e38f)) atomicOr(p.status, 1);
            collide_store<1>(q, o.self(), g, m, [&](auto ic, float gi) {
                return transport<1, MODE, decltype(ic)::value, 2>(q, o, gi);
            });
            if (ROT) {
                float adv[7];
                rot_advect<1, 2>(q, o, h, m, adv);
                rot_store(q, o.self(), h, m, adv);
            }
            if (has_left && l < 3) {
                float *far = cluster.map_shared_rank(b, left);
#pragma unroll
                for (int i = 0; i < POPS; ++i) far[i * pitch + n_left + 3 + l] = b[i * pitch + l + 3];
            }
            if (has_right && l >= n - 3) {
                float *far = cluster.map_shared_rank(b, right);
#pragma unroll
                for (int i = 0; i < POPS; ++i) far[i * pitch + l - (n - 3)] = b[i * pitch + l + 3];
            }
        }
        float *t = a;
        a = b;
        b = t;
        cluster.sync();  // step s + 1 reads what the neighbours wrote, and may overwrite what they read
    }
    if (l < n) {
#pragma unroll
        for (int i = 0; i < POPS; ++i) p.dst[(size_t)i * p.S + c0 + l] = a[i * pitch + l + 3];
    }
}

template <bool ROT, int MODE, int MAXT> cudaError_t launch_tube_t(const Args &a, int64_t steps, cudaStream_t s)
{
    const auto p = make_params<7, float>(a);
    // as many blocks as leave each at least a warp of nodes
    const int blocks = std::min(kTubeCluster, std::max(1, a.X / kTubeMinPiece));
    const int piece = (a.X + blocks - 1) / blocks;
    const int pitch = piece + 6;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3((piece + 31) / 32 * 32);
    cfg.dynamicSmemBytes = sizeof(float) * 2 * (ROT ? 14 : 7) * pitch;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = blocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cfg.dynamicSmemBytes > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k_tube_steps<ROT, MODE, MAXT>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)cfg.dynamicSmemBytes);
        if (e != cudaSuccess) return e;
    }
    return cudaLaunchKernelEx(&cfg, k_tube_steps<ROT, MODE, MAXT>, p, steps, pitch);
}

template <bool ROT, int MODE> cudaError_t launch_tube(const Args &a, int64_t steps, cudaStream_t s)
{
    return a.X <= kTubeCluster * 256 ? launch_tube_t<ROT, MODE, 256>(a, steps, s)
                                     : launch_tube_t<ROT, MODE, kTubeMaxPiece>(a, steps, s);
}

}  // namespace

// Whether `steps` steps of this problem run as one launch: float storage, a
// tube whose pieces fit one node a thread (8192 nodes, where a block of 1024
// threads still takes less than the launch and eight times the blocks gain
// little), long enough for a halo beside every piece, and enough steps to pay for
// loading and storing the state.
bool tube_steps_ok(const Args &a, int64_t steps)
{
    return a.storage == 0 && a.X >= kTubeMinPiece && a.X <= kTubeCluster * kTubeMaxPiece && steps >= 4;
}

cudaError_t launch_tube_steps(const Args &a, int64_t steps, cudaStream_t s)
{
    if (a.Qr > 0) return a.mode ? launch_tube<true, 1>(a, steps, s) : launch_tube<true, 0>(a, steps, s);
    return a.mode ? launch_tube<false, 1>(a, steps, s) : launch_tube<false, 0>(a, steps, s);
}

cudaError_t launch_d1q7(Op op, const Args &a, cudaStream_t s) { return launch_lattice<1>(op, a, s); }
}  // namespace lbm
