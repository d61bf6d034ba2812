// Ensembles of independent 1-D problems (D1Q7 + D1Q7, copy ends) advanced
// by one persistent launch: the lbm_batch_* part of the C ABI (include/lbm.h).
//
// Each resident block claims whole problems, longest first, from an atomic
// counter and runs all k steps of its problem; the node update is
// lbm_step's (lbm_tube.cuh), so results are bit-identical to running each
// problem alone.  A per-problem watch range limits which nodes may set its
// status word.
#include <algorithm>
#include <cmath>
#include <numeric>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/lbm.h"
#include "lbm_tube.cuh"

namespace lbm {
namespace {

constexpr int kD1 = 1;  // Lattice<1> = D1Q7

struct TubeDesc {    // one problem, indexed by its original position
    uint32_t base;   // first float of the problem in a state buffer
    int len;         // nodes
    int pitch;       // floats per population array (len rounded up to 32)
    int node_off;    // first node in the macro arrays
    float omega;     // BGK rate, with 1 - omega exact in float
    float cT;        // (D + n)/2
    float half_n;    // n/2
    float half_n_r2; // n r^2 / 2
    int watch_lo;    // nodes [watch_lo, watch_hi) set the status word
    int watch_hi;
};

struct BatchParams {
    const TubeDesc *tubes;
    const int *order;  // processing order (longest first)
    int count;
    float *buf[2];
    int cur;           // buffer holding the state at step 0
    long long steps;
    int *status;       // per problem
    int *counter;
    float r, r2, inv_r2, nu_scale, inv_m;
    float w[7], wr[7];
};

__device__ __forceinline__ Params<7> tube_params(const BatchParams &bp, const TubeDesc &d,
                                                 const float *src, float *dst)
{
    Params<7> p;
    p.src = src ? src + d.base : nullptr;
    p.dst = dst ? dst + d.base : nullptr;
    p.in0 = p.in1 = p.in2 = nullptr;
    p.out0 = p.out1 = p.out2 = nullptr;
    p.status = nullptr;
    p.partials = nullptr;
    p.S = d.pitch;
    p.N = d.len;
    p.X = d.len;
    p.Y = 1;
    p.Z = 1;
    p.pitch = d.pitch;
    p.bc0 = LBM_BC_COPY;
    p.bc1 = p.bc2 = LBM_BC_PERIODIC;
    p.r = bp.r;
    p.r2 = bp.r2;
    p.inv_r2 = bp.inv_r2;
    p.omega = d.omega;
    p.nu_scale = bp.nu_scale;
    p.cT = d.cT;
    p.half_n = d.half_n;
    p.half_n_r2 = d.half_n_r2;
    p.inv_m = bp.inv_m;
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        p.w[i] = bp.w[i];
        p.wr[i] = bp.wr[i];
    }
    return p;
}

// The state of the nodes a block works on lies in shared memory, two copies,
// node by node and 15 floats apart: every population and neighbour is an
// immediate offset from one address (a third of the instructions of the
// population-major form were address arithmetic), and the odd pitch keeps
// consecutive lanes on different banks.  A thread updates one node at a time,
// with a block barrier between steps; the new state is stored after the last
// load, and an end's thread stores its node's three copies beyond the end from
// registers.
//
// A problem that fits (kWindow nodes, 108 KB: two blocks an SM) is loaded once
// and stored after its last step.  A longer one goes through the two global
// buffers in passes of at most kPassSteps steps: a pass loads each window of
// the problem with as many nodes beside it as the steps can reach (two a step,
// three in STREAM mode), runs them, and stores the window's inside, which is
// exactly what whole steps give; the nodes beside it go wrong from the
// window's ends inwards and are dropped.  Against one pass over the global
// buffers per step this reads and writes L2 once in sixteen steps, for 8-12 %
// more nodes.
//
// Bound by issue (81 % of the slots at 1024 x 384 nodes), shared-memory reads (LSU
// 63 %) and the barriers between steps.  One node a
// thread against two in packed arithmetic (f32x2, half a window apart), 32 FD
// steps: 1024 tubes of 4096 nodes 1.78 / 2.01 ms, of 640 285 / 335 us, of 384 179
// / 172, of 100-150 83 / 102; 152 tubes of 384 41 / 54, one of 100-150 30 / 45: a
// step of a short problem is one node's chain of instructions.  Copying the end's
// node through shared memory, value by value, made that chain 0.5 us longer.
// 1024 tubes of 256-8192 nodes, 50 FD steps 3.12 ms (6.53 through the global
// buffers); passes of 8 / 12 / 16 steps and windows of 448 / 896 nodes, two nodes
// a thread: 3.66 / 3.52 / 3.43 and 3.84 / 3.43.
constexpr int kNodePitch = 15;
#ifndef LBM_BATCH_WINDOW
#define LBM_BATCH_WINDOW 896
#endif
#ifndef LBM_BATCH_PASS
#define LBM_BATCH_PASS 16
#endif
constexpr int kWindow = LBM_BATCH_WINDOW;
constexpr int kPassSteps = LBM_BATCH_PASS;
#ifndef LBM_BATCH_THREADS
#define LBM_BATCH_THREADS 512
#endif

template <int MODE>
__global__ void __launch_bounds__(1024) k_batch_run(const BatchParams bp, const TubeLattice lat, int nodes)
{
    extern __shared__ float sm[];  // [2][nodes][kNodePitch]
    __shared__ int claim;
    constexpr int kReach = MODE ? 2 : 3;
    for (;;) {
        if (threadIdx.x == 0) claim = atomicAdd(bp.counter, 1);
        __syncthreads();
        const int slot = claim;
        __syncthreads();  // every thread has read `claim` before it is reused
        if (slot >= bp.count) return;
        const int k = bp.order[slot];
        const TubeDesc d = bp.tubes[k];
        const TubeRates rates = tube_rates(d.omega, d.cT, d.half_n);
        // passes: one if the problem fits, else enough of them for the longest
        // to be kPassSteps and their parity that of the steps, which decides
        // the buffer the caller expects the state in
        const bool fits = d.len <= nodes - 6;
        int64_t passes = 1;
        if (!fits) {
            passes = (bp.steps + kPassSteps - 1) / kPassSteps;
            passes += (passes ^ bp.steps) & 1;
        }
        const int halo = fits ? 0 : kReach * kPassSteps;
        const int windows = fits ? 1 : (d.len + (nodes - 6 - 2 * halo) - 1) / (nodes - 6 - 2 * halo);
        int cur = bp.cur;
        for (int64_t q = 0; q < passes; ++q) {
            const int64_t steps = bp.steps * (q + 1) / passes - bp.steps * q / passes;
            const int end = fits ? bp.cur ^ (int)(bp.steps & 1) : cur ^ 1;
            const float *in = bp.buf[cur] + d.base;
            float *out = bp.buf[end] + d.base;
            for (int wi = 0; wi < windows; ++wi) {
                const int i0 = (int)((int64_t)d.len * wi / windows), i1 = (int)((int64_t)d.len * (wi + 1) / windows);
                const int w0 = max(0, i0 - halo), w1 = min(d.len, i1 + halo), n = w1 - w0;
                float *a = sm, *c = sm + nodes * kNodePitch;
                // local node l + 3 is node w0 + l; the ends' copies, and
                // nothing to rely on beyond a window's inner end
                for (int l = threadIdx.x; l < n + 6; l += blockDim.x) {
                    const int x = min(max(w0 + l - 3, 0), d.len - 1);
#pragma unroll
                    for (int i = 0; i < 14; ++i) a[l * kNodePitch + i] = __ldcg(in + (uint32_t)(i * d.pitch + x));
                }
                __syncthreads();
                const bool left = w0 == 0, right = w1 == d.len;
                const int watch_lo = max(i0, d.watch_lo), watch_hi = min(i1, d.watch_hi);
                for (int64_t s = 0; s < steps; ++s) {
                    for (int l = threadIdx.x; l < n; l += blockDim.x) {
                        const float *me = a + (l + 3) * kNodePitch;
                        float out[14], rho, T;
                        tube_update<true, MODE>(
                            lat, rates, [&](int pop, int dx) { return me[dx * kNodePitch + pop]; },
                            [&](float ux) {
                                const int up = ux >= 0.f ? -kNodePitch : kNodePitch;
                                const float *u1 = me + up, *u2 = me + 2 * up, *d1 = me - up;
                                return [u1, u2, d1](int j, int kk) { return (kk == 2 ? u2 : kk == 1 ? u1 : d1)[7 + j]; };
                            },
                            out, rho, T);
                        if (tube_bad(rho, T) && w0 + l >= watch_lo && w0 + l < watch_hi) atomicOr(bp.status + k, 1);
                        auto put = [&](int at) {
#pragma unroll
                            for (int i = 0; i < 14; ++i) c[at * kNodePitch + i] = out[i];
                        };
                        put(l + 3);
                        // the copies beyond the problem's ends
                        if (left && l == 0) {
#pragma unroll 1
                            for (int g = 0; g < 3; ++g) put(g);
                        }
                        if (right && l == n - 1) {
#pragma unroll 1
                            for (int g = 0; g < 3; ++g) put(n + 3 + g);
                        }
                    }
                    float *t = a;
                    a = c;
                    c = t;
                    __syncthreads();  // step s + 1 reads neighbours written in step s
                }
                for (int l = threadIdx.x; l < i1 - i0; l += blockDim.x) {
#pragma unroll
                    for (int i = 0; i < 14; ++i)
                        out[(uint32_t)(i * d.pitch + i0 + l)] = a[(i0 - w0 + l + 3) * kNodePitch + i];
                }
                __syncthreads();  // the window's state has been read; its stores precede the next pass
            }
            cur = end;
        }
    }
}

template <int MODE>
__global__ void __launch_bounds__(kBlockX) k_batch_init(const BatchParams bp, const float *rho,
                                                        const float *u, const float *T)
{
    const TubeDesc d = bp.tubes[blockIdx.y];
    const int x = blockIdx.x * kBlockX + threadIdx.x;
    if (x >= d.len) return;
    Params<7> p = tube_params(bp, d, nullptr, bp.buf[bp.cur]);
    p.in0 = rho + d.node_off;
    p.in1 = u + d.node_off;
    p.in2 = T + d.node_off;
    init_node<kD1, true, MODE>(p, x, 0, 0);
}

template <int MODE>
__global__ void __launch_bounds__(kBlockX) k_batch_moments(const BatchParams bp, float *rho,
                                                           float *u, float *T)
{
    const TubeDesc d = bp.tubes[blockIdx.y];
    const int x = blockIdx.x * kBlockX + threadIdx.x;
    if (x >= d.len) return;
    Params<7> p = tube_params(bp, d, bp.buf[bp.cur], nullptr);
    p.out0 = rho + d.node_off;
    p.out1 = u + d.node_off;
    p.out2 = T + d.node_off;
    moments_node<kD1, true, MODE>(p, x, 0, 0);
}

// D1Q7 constants solved in double precision (lbm_lattice_info).
void d1q7(double *r, double w[7])
{
    int e[343 * 3];
    lbm_lattice_info(LBM_D1Q7, r, e, w);
}

size_t align256(size_t n) { return (n + 255) / 256 * 256; }

}  // namespace
}  // namespace lbm

using lbm::BatchParams;
using lbm::TubeDesc;

struct lbm_batch_ctx {
    int count = 0, mode = LBM_MODE_STREAM, m_fd = 1;
    double r = 0.0, w[7] = {};
    std::vector<TubeDesc> tubes;
    std::vector<int> order;
    int max_len = 0;
    int window = 0;    // nodes a block's shared memory holds, six of them beyond the ends
    int64_t total_nodes = 0;
    size_t state_floats = 0;
    size_t off_tubes = 0, off_order = 0, off_status = 0, off_counter = 0, work_bytes = 0;
    bool bound = false, has_state = false;
    float *buf[2] = {nullptr, nullptr};
    char *work = nullptr;
    cudaStream_t stream = nullptr;
    int cur = 0;
    int threads = LBM_BATCH_THREADS;  // threads per block at most, a node each
    int blocks_per_sm = 0;            // resident blocks per SM of the persistent grid (0 = max)
    int64_t launches = 0;
    std::string err;
    struct Cached {
        cudaGraphExec_t exec = nullptr;
        long long steps = -1;
        int cur = -1, threads = -1, bps = -1;
    } graphs[2];
    int next_graph = 0;
};

namespace {

int bfail(lbm_batch b, int code, const std::string &msg)
{
    if (b) b->err = msg;
    return code;
}

int bcuda(lbm_batch b, cudaError_t e, const char *where)
{
    return bfail(b, LBM_ECUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

BatchParams batch_params(const lbm_batch_ctx *b, long long steps)
{
    BatchParams bp{};
    bp.tubes = reinterpret_cast<const TubeDesc *>(b->work + b->off_tubes);
    bp.order = reinterpret_cast<const int *>(b->work + b->off_order);
    bp.count = b->count;
    bp.buf[0] = b->buf[0];
    bp.buf[1] = b->buf[1];
    bp.cur = b->cur;
    bp.steps = steps;
    bp.status = reinterpret_cast<int *>(b->work + b->off_status);
    bp.counter = reinterpret_cast<int *>(b->work + b->off_counter);
    const double m = (b->mode == LBM_MODE_FD) ? b->m_fd : 1.0;
    bp.r = (float)b->r;
    bp.r2 = bp.r * bp.r;
    bp.inv_r2 = 1.0f / (bp.r * bp.r);
    bp.nu_scale = (float)(1.0 / (m * b->r));
    bp.inv_m = (float)(1.0 / m);
    for (int j = 0; j < 7; ++j) {
        bp.w[j] = (float)b->w[j];
        bp.wr[j] = (float)b->w[j];
    }
    return bp;
}

bool aligned(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 255u) == 0; }

// The persistent kernel of a run, its threads and its dynamic shared memory.
const void *run_kernel(const lbm_batch_ctx *b)
{
    return (b->mode == LBM_MODE_FD) ? (const void *)lbm::k_batch_run<1> : (const void *)lbm::k_batch_run<0>;
}
// No more threads than a window has nodes: the others would take registers from
// other blocks (1024 tubes of 100-150 nodes, two nodes a thread: 108 us with as
// many as needed, 145 with 256).  Windows of 257 to 512 nodes, from three problems per SM on: 256
// threads, which four blocks an SM can have: 600 / 1024 / 3000 problems of 450-512
// nodes 127 / 217 / 571 us against 164 / 229 / 618 with a node a thread; 300 / 450
// problems 76 / 103 against 75 / 102.
int run_threads(const lbm_batch_ctx *b, int threads, int sms)
{
    const int nodes = (b->window - 6 + 31) / 32 * 32;
    const int most = nodes > 256 && nodes <= 512 && b->count > 3 * sms ? 256 : nodes;
    return std::min(threads, most);
}
int run_smem(const lbm_batch_ctx *b) { return (int)sizeof(float) * 2 * lbm::kNodePitch * b->window; }

// Threads per block and grid of the persistent kernel.
cudaError_t persistent_grid(const lbm_batch_ctx *b, int threads, int bps, int *block, int *grid)
{
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const void *fn = run_kernel(b);
    *block = run_threads(b, threads, sms);
    // (the limit is a property of the kernel, which other ensembles share: the
    // largest any of them takes)
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(float) * 2 * lbm::kNodePitch * (lbm::kWindow + 6));
    if (e == cudaSuccess)  // all of L1 as shared memory: the kernel reads nothing twice through it
        e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, *block, run_smem(b));
    if (e != cudaSuccess) return e;
    per_sm = std::max(1, per_sm);
    if (bps > 0) per_sm = std::min(per_sm, bps);
    // (a block per problem at most: more would claim unevenly, several problems
    // on some SMs while others have none)
    *grid = std::min(per_sm * sms, b->count);
    return cudaSuccess;
}

// The graph of one run: reset the claim counter, then the persistent kernel.
int build_graph(lbm_batch b, long long steps, cudaGraphExec_t *exec)
{
    int block = 0, grid = 0;
    cudaError_t e = persistent_grid(b, b->threads, b->blocks_per_sm, &block, &grid);
    if (e != cudaSuccess) return bcuda(b, e, "occupancy query");
    cudaGraph_t g = nullptr;
    e = cudaGraphCreate(&g, 0);
    if (e != cudaSuccess) return bcuda(b, e, "cudaGraphCreate");
    cudaMemsetParams ms{};
    ms.dst = b->work + b->off_counter;
    ms.value = 0;
    ms.elementSize = 4;
    ms.width = 1;
    ms.height = 1;
    ms.pitch = 4;
    cudaGraphNode_t n_reset = nullptr, n_run = nullptr;
    e = cudaGraphAddMemsetNode(&n_reset, g, nullptr, 0, &ms);
    BatchParams bp = batch_params(b, steps);
    lbm::TubeLattice lat = lbm::tube_lattice(bp.w, bp.r, bp.nu_scale, bp.inv_m);
    int window = b->window;
    void *args[] = {&bp, &lat, &window};
    cudaKernelNodeParams kp{};
    kp.func = const_cast<void *>(run_kernel(b));
    kp.gridDim = dim3(grid);
    kp.blockDim = dim3(block);
    kp.sharedMemBytes = (unsigned)run_smem(b);
    kp.kernelParams = args;
    if (e == cudaSuccess) e = cudaGraphAddKernelNode(&n_run, g, &n_reset, 1, &kp);
    if (e == cudaSuccess) e = cudaGraphInstantiate(exec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return bcuda(b, e, "graph build");
    return LBM_OK;
}

}  // namespace

extern "C" {

int lbm_batch_create(int count, const int64_t *lengths, const int *n, const double *tau, int mode,
                     int m_fd, lbm_batch *out)
{
    if (!out) return LBM_EINVAL;
    *out = nullptr;
    if (count < 1 || count > 65535 || !lengths || !n || !tau) return LBM_EINVAL;
    if (mode != LBM_MODE_STREAM && mode != LBM_MODE_FD) return LBM_EINVAL;
    if (mode == LBM_MODE_FD && m_fd < 1) return LBM_EINVAL;
    lbm_batch b = new lbm_batch_ctx();
    b->count = count;
    b->mode = mode;
    b->m_fd = (mode == LBM_MODE_FD) ? m_fd : 1;
    lbm::d1q7(&b->r, b->w);
    const double m = b->m_fd;
    b->tubes.resize(count);
    size_t base = 0;
    int64_t node = 0;
    for (int k = 0; k < count; ++k) {
        if (lengths[k] < 1 || lengths[k] > (1 << 30) || n[k] < 0 || !(tau[k] > 0.0) ||
            !std::isfinite(tau[k])) {
            delete b;
            return LBM_EINVAL;
        }
        TubeDesc &d = b->tubes[k];
        d.len = (int)lengths[k];
        d.pitch = (d.len + 31) / 32 * 32;
        d.base = (uint32_t)base;
        d.node_off = (int)node;
        // omega with an exact 1 - omega, as for lbm_handle
        const float om = (float)(1.0 / (m * tau[k]));
        const float keep = (float)(1.0 - (double)om);
        d.omega = (float)(1.0 - (double)keep);
        d.cT = (float)(0.5 * (1 + n[k]));
        d.half_n = (float)(0.5 * n[k]);
        d.half_n_r2 = (float)(0.5 * n[k] * b->r * b->r);
        d.watch_lo = 0;
        d.watch_hi = d.len;
        base += (size_t)14 * d.pitch;
        node += d.len;
        b->max_len = std::max(b->max_len, d.len);
        if (base > 0x7fffffffULL || node > 0x7fffffffLL) {
            delete b;
            return LBM_ESIZE;
        }
    }
    b->state_floats = base;
    b->total_nodes = node;
    b->window = std::min(b->max_len, lbm::kWindow) + 6;
    b->order.resize(count);
    std::iota(b->order.begin(), b->order.end(), 0);
    std::stable_sort(b->order.begin(), b->order.end(),
                     [&](int a, int c) { return b->tubes[a].len > b->tubes[c].len; });
    b->off_tubes = 0;
    b->off_order = lbm::align256(sizeof(TubeDesc) * count);
    b->off_status = b->off_order + lbm::align256(sizeof(int) * count);
    b->off_counter = b->off_status + lbm::align256(sizeof(int) * count);
    b->work_bytes = b->off_counter + 256;
    *out = b;
    return LBM_OK;
}

int lbm_batch_set_problems(lbm_batch b, const int *n, const double *tau)
{
    if (!b) return LBM_EINVAL;
    if (!n || !tau) return bfail(b, LBM_EINVAL, "null n or tau");
    for (int k = 0; k < b->count; ++k)
        if (n[k] < 0 || !(tau[k] > 0.0) || !std::isfinite(tau[k]))
            return bfail(b, LBM_EINVAL, "bad n or tau");
    const double m = b->m_fd;
    for (int k = 0; k < b->count; ++k) {
        TubeDesc &d = b->tubes[k];
        const float om = (float)(1.0 / (m * tau[k]));
        const float keep = (float)(1.0 - (double)om);
        d.omega = (float)(1.0 - (double)keep);
        d.cT = (float)(0.5 * (1 + n[k]));
        d.half_n = (float)(0.5 * n[k]);
        d.half_n_r2 = (float)(0.5 * n[k] * b->r * b->r);
    }
    if (b->bound) {
        cudaError_t e = cudaMemcpyAsync(b->work + b->off_tubes, b->tubes.data(),
                                        sizeof(TubeDesc) * b->count, cudaMemcpyHostToDevice,
                                        b->stream);
        if (e != cudaSuccess) return bcuda(b, e, "table upload");
        b->has_state = false;
    }
    return LBM_OK;
}

int lbm_batch_set_watch(lbm_batch b, const int *lo, const int *hi)
{
    if (!b) return LBM_EINVAL;
    if ((lo == nullptr) != (hi == nullptr)) return bfail(b, LBM_EINVAL, "lo and hi go together");
    for (int k = 0; lo && k < b->count; ++k)
        if (lo[k] < 0 || lo[k] > hi[k] || hi[k] > b->tubes[k].len)
            return bfail(b, LBM_EINVAL, "watch range outside the problem");
    for (int k = 0; k < b->count; ++k) {
        b->tubes[k].watch_lo = lo ? lo[k] : 0;
        b->tubes[k].watch_hi = lo ? hi[k] : b->tubes[k].len;
    }
    if (b->bound) {
        cudaError_t e = cudaMemcpyAsync(b->work + b->off_tubes, b->tubes.data(),
                                        sizeof(TubeDesc) * b->count, cudaMemcpyHostToDevice,
                                        b->stream);
        if (e != cudaSuccess) return bcuda(b, e, "table upload");
    }
    return LBM_OK;
}

int lbm_batch_sizes(lbm_batch b, size_t *state_bytes, size_t *work_bytes, int64_t *total_nodes)
{
    if (!b) return LBM_EINVAL;
    if (state_bytes) *state_bytes = sizeof(float) * b->state_floats;
    if (work_bytes) *work_bytes = b->work_bytes;
    if (total_nodes) *total_nodes = b->total_nodes;
    return LBM_OK;
}

int lbm_batch_bind(lbm_batch b, void *buf_a, void *buf_b, size_t state_bytes, void *work,
                   size_t work_bytes, void *stream)
{
    if (!b) return LBM_EINVAL;
    if (!buf_a || !buf_b || !work || buf_a == buf_b) return bfail(b, LBM_EINVAL, "bad buffers");
    if (!aligned(buf_a) || !aligned(buf_b) || !aligned(work))
        return bfail(b, LBM_EINVAL, "buffers must be 256-byte aligned");
    if (state_bytes < sizeof(float) * b->state_floats || work_bytes < b->work_bytes)
        return bfail(b, LBM_ESIZE, "buffer smaller than reported by lbm_batch_sizes");
    b->buf[0] = static_cast<float *>(buf_a);
    b->buf[1] = static_cast<float *>(buf_b);
    b->work = static_cast<char *>(work);
    b->stream = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaMemcpyAsync(b->work + b->off_tubes, b->tubes.data(),
                                    sizeof(TubeDesc) * b->count, cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(b->work + b->off_order, b->order.data(), sizeof(int) * b->count,
                            cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(b->work + b->off_status, 0, sizeof(int) * b->count, b->stream);
    if (e != cudaSuccess) return bcuda(b, e, "table upload");
    for (auto &c : b->graphs) {
        if (c.exec) cudaGraphExecDestroy(c.exec);
        c = lbm_batch_ctx::Cached{};
    }
    b->bound = true;
    b->has_state = false;
    b->cur = 0;
    return LBM_OK;
}

int lbm_batch_set_macro(lbm_batch b, const float *rho, const float *u, const float *T)
{
    if (!b) return LBM_EINVAL;
    if (!b->bound) return bfail(b, LBM_ESTATE, "lbm_batch_bind must precede lbm_batch_set_macro");
    if (!rho || !u || !T) return bfail(b, LBM_EINVAL, "null field pointer");
    b->cur = 0;
    BatchParams bp = batch_params(b, 0);
    const dim3 grid((b->max_len + lbm::kBlockX - 1) / lbm::kBlockX, b->count);
    if (b->mode == LBM_MODE_FD)
        lbm::k_batch_init<1><<<grid, lbm::kBlockX, 0, b->stream>>>(bp, rho, u, T);
    else
        lbm::k_batch_init<0><<<grid, lbm::kBlockX, 0, b->stream>>>(bp, rho, u, T);
    ++b->launches;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaMemsetAsync(b->work + b->off_status, 0, sizeof(int) * b->count, b->stream);
    if (e != cudaSuccess) return bcuda(b, e, "batch init");
    b->has_state = true;
    return LBM_OK;
}

int lbm_batch_run(lbm_batch b, int64_t k)
{
    if (!b) return LBM_EINVAL;
    if (k < 0) return bfail(b, LBM_EINVAL, "k must be >= 0");
    if (!b->has_state) return bfail(b, LBM_ESTATE, "no state: call lbm_batch_set_macro");
    if (k == 0) return LBM_OK;
    lbm_batch_ctx::Cached *hit = nullptr;
    for (auto &c : b->graphs)
        if (c.exec && c.steps == k && c.cur == b->cur && c.threads == b->threads &&
            c.bps == b->blocks_per_sm)
            hit = &c;
    if (!hit) {
        hit = &b->graphs[b->next_graph];
        b->next_graph ^= 1;
        if (hit->exec) cudaGraphExecDestroy(hit->exec);
        *hit = lbm_batch_ctx::Cached{};
        const int rc = build_graph(b, k, &hit->exec);
        if (rc != LBM_OK) return rc;
        hit->steps = k;
        hit->cur = b->cur;
        hit->threads = b->threads;
        hit->bps = b->blocks_per_sm;
    }
    cudaError_t e = cudaGraphLaunch(hit->exec, b->stream);
    if (e != cudaSuccess) return bcuda(b, e, "cudaGraphLaunch");
    ++b->launches;
    b->cur ^= (int)(k & 1);
    return LBM_OK;
}

int lbm_batch_get_moments(lbm_batch b, float *rho, float *u, float *T)
{
    if (!b) return LBM_EINVAL;
    if (!b->has_state) return bfail(b, LBM_ESTATE, "no state");
    if (!rho || !u || !T) return bfail(b, LBM_EINVAL, "null field pointer");
    BatchParams bp = batch_params(b, 0);
    const dim3 grid((b->max_len + lbm::kBlockX - 1) / lbm::kBlockX, b->count);
    if (b->mode == LBM_MODE_FD)
        lbm::k_batch_moments<1><<<grid, lbm::kBlockX, 0, b->stream>>>(bp, rho, u, T);
    else
        lbm::k_batch_moments<0><<<grid, lbm::kBlockX, 0, b->stream>>>(bp, rho, u, T);
    ++b->launches;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return bcuda(b, e, "batch moments");
    return LBM_OK;
}

int lbm_batch_status(lbm_batch b, int *status, int *n_bad)
{
    if (!b) return LBM_EINVAL;
    if (!b->bound) return bfail(b, LBM_ESTATE, "not bound");
    std::vector<int> host(b->count);
    cudaError_t e = cudaMemcpyAsync(host.data(), b->work + b->off_status, sizeof(int) * b->count,
                                    cudaMemcpyDeviceToHost, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return bcuda(b, e, "status readback");
    int bad = 0;
    for (int k = 0; k < b->count; ++k) bad += host[k] != 0;
    if (status) std::copy(host.begin(), host.end(), status);
    if (n_bad) *n_bad = bad;
    return LBM_OK;
}

int lbm_batch_set_block(lbm_batch b, int threads, int blocks_per_sm)
{
    if (!b) return LBM_EINVAL;
    if (threads < 32 || threads > 1024 || threads % 32)
        return bfail(b, LBM_EINVAL, "threads must be a multiple of 32 in 32..1024");
    if (blocks_per_sm < 0) return bfail(b, LBM_EINVAL, "blocks_per_sm must be >= 0");
    b->threads = threads;
    b->blocks_per_sm = blocks_per_sm;
    return LBM_OK;
}

int lbm_batch_autotune(lbm_batch b, int64_t sample_steps, int *threads, int *blocks_per_sm)
{
    if (!b) return LBM_EINVAL;
    if (sample_steps < 1) return bfail(b, LBM_EINVAL, "sample_steps must be >= 1");
    if (!b->has_state) return bfail(b, LBM_ESTATE, "no state: call lbm_batch_set_macro");
    // Block size x resident blocks per SM: fewer resident problems keep more
    // of each one's state in L2, more blocks hide more latency.
    static const int cand_threads[] = {128, 256, 512, 1024};
    static const int cand_bps[] = {1, 2, 4, 0};
    cudaEvent_t t0, t1;
    cudaError_t e = cudaEventCreate(&t0);
    if (e == cudaSuccess) e = cudaEventCreate(&t1);
    if (e != cudaSuccess) return bcuda(b, e, "cudaEventCreate");
    float best_ms = 0.f;
    int best_t = b->threads, best_b = b->blocks_per_sm;
    for (int c : cand_threads) {
        for (int bps : cand_bps) {
            b->threads = c;
            b->blocks_per_sm = bps;
            int rc = lbm_batch_run(b, sample_steps);  // builds the graph, warms up
            if (rc != LBM_OK) break;
            e = cudaEventRecord(t0, b->stream);
            rc = lbm_batch_run(b, sample_steps);
            if (rc != LBM_OK) break;
            if (e == cudaSuccess) e = cudaEventRecord(t1, b->stream);
            if (e == cudaSuccess) e = cudaEventSynchronize(t1);
            float ms = 0.f;
            if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, t0, t1);
            if (e != cudaSuccess) break;
            if (best_ms == 0.f || ms < best_ms) {
                best_ms = ms;
                best_t = c;
                best_b = bps;
            }
        }
        if (e != cudaSuccess) break;
    }
    cudaEventDestroy(t0);
    cudaEventDestroy(t1);
    b->threads = best_t;
    b->blocks_per_sm = best_b;
    if (threads) *threads = best_t;
    if (blocks_per_sm) *blocks_per_sm = best_b;
    if (e != cudaSuccess) return bcuda(b, e, "autotune timing");
    return LBM_OK;
}

int64_t lbm_batch_launch_count(lbm_batch b) { return b ? b->launches : -1; }

const char *lbm_batch_last_error(lbm_batch b) { return b ? b->err.c_str() : "null handle"; }

void lbm_batch_destroy(lbm_batch b)
{
    if (!b) return;
    for (auto &c : b->graphs)
        if (c.exec) cudaGraphExecDestroy(c.exec);
    delete b;
}

}  // extern "C"
