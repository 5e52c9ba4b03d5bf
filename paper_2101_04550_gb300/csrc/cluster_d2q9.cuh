// Several time steps of a small D2Q9 grid in one launch.
//
// A step of a few thousand nodes is all latency: one launch per step of the row march
// (single_pass_d2q9.cuh) spends 4.1 us on a 64 x 64 grid, most of it the chain of row
// loads and the launch.  Here one thread-block cluster keeps the whole grid in the
// shared memory of its (up to 8) blocks and advances it nsteps steps: a block owns a
// band of rows, its populations twice (source and destination) and their anomaly.
// Per step
//   * every node's moments and anomaly (Eqs. density, momentum, Deviation); Q~_yyy of
//     a band's first and last row also goes to the neighbouring block (distributed
//     shared memory), then the cluster's barrier;
//   * relaxation (Eqs. Paastar1, 27eqext, LBGK) and the push to (x + cx, y + cy) of
//     the destination, the rows beyond the band into the neighbouring block, then
//     the cluster's barrier.
// The per-node arithmetic is the row march's (moments_of, anomaly, relax_streamed),
// and values are rounded to the storage type in shared memory as they are in the
// population array, so the results agree bit for bit.
//
// Bound by the two barriers and the dependent chain of a step: 1.55 us at 64 x 64 (one
// node a thread; 1.85 with its populations and moments read again after the barrier).
#pragma once
#include <cooperative_groups.h>

#include "single_pass_d2q9.cuh"

namespace elbm {

constexpr int kClThreads = 512;
constexpr int kClBlocks = 8;        // blocks of the cluster at most (the portable size)
constexpr int kClMaxSteps = 4096;   // steps of one launch at most

template <int ST>
__global__ void __launch_bounds__(kClThreads, 1)
    k_cluster_d2q9(const __grid_constant__ StepParams p, int band, int nsteps)
{
    using S = Storage<ST>;
    using T = typename S::T;
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nx = p.nx, rank = (int)cluster.block_rank(), ranks = (int)cluster.num_blocks();
    const int row0 = rank * band, rows = min(band, p.ny - row0), nodes = rows * nx;
    const int below = rank == 0 ? ranks - 1 : rank - 1, above = rank == ranks - 1 ? 0 : rank + 1;
    const int rows_below = min(band, p.ny - below * band);
    // qx[band][nx], qy[band + 2][nx] (a row more at either end), populations [2][9][band][nx]
    float* qx = reinterpret_cast<float*>(smem_raw);
    float* qy = qx + band * nx;
    T* pops = reinterpret_cast<T*>(qy + (band + 2) * nx);
    const int plane = band * nx;  // stride between populations
    float* qy_below = cluster.map_shared_rank(qy, below) + (rows_below + 1) * nx;  // its row above the last
    float* qy_above = cluster.map_shared_rank(qy, above);                          // its row below the first
    T* f = static_cast<T*>(p.f);

    for (int t = threadIdx.x; t < nodes; t += kClThreads)
#pragma unroll
        for (int i = 0; i < 9; ++i) pops[i * plane + t] = f[i * p.N + row0 * nx + t];
    cluster.sync();  // every block runs and holds its band

    int cur = 0;
    for (int step = 0; step < nsteps; ++step) {
        const T* src = pops + cur * 9 * plane;
        T* dst = pops + (cur ^ 1) * 9 * plane;
        T* dst_below = cluster.map_shared_rank(dst, below) + (rows_below - 1) * nx;  // its last row
        T* dst_above = cluster.map_shared_rank(dst, above);                          // its first row
        // populations and moments of a thread's first node stay in registers over the
        // barrier; it reads those of further ones again
        float g0[9], drho0 = 0.f, j0[3] = {0.f, 0.f, 0.f}, inv0 = 1.f;
        auto load = [&](int t, float* g, float& drho, float* j, float& inv) {
#pragma unroll
            for (int i = 0; i < 9; ++i) g[i] = raw_value<ST>(p, src[i * plane + t], i);
            moments_of<2>(p, [&](int i) { return g[i]; }, drho, j);
            inv = 1.0f / (p.rho_ref + drho);
        };
        auto publish = [&](int t, const float* j, float inv) {
            qx[t] = anomaly(p, 0, j[0], j[0] * inv);
            const float q = anomaly(p, 1, j[1], j[1] * inv);
            qy[nx + t] = q;
            if (t < nx) qy_below[t] = q;
            if (t >= nodes - nx) qy_above[t - (nodes - nx)] = q;
        };
        if (threadIdx.x < nodes) {
            load(threadIdx.x, g0, drho0, j0, inv0);
            publish(threadIdx.x, j0, inv0);
        }
        for (int t = threadIdx.x + kClThreads; t < nodes; t += kClThreads) {
            float g[9], drho, j[3], inv;
            load(t, g, drho, j, inv);
            publish(t, j, inv);
        }
        cluster.sync();
        auto relax_node = [&](int t, const float* g, float drho, const float* j, float inv) {
            const int y = fast_div(t, p.div_nx_m, p.div_nx_s), x = t - y * nx;
            const int xo[3] = {x == 0 ? nx - 1 : x - 1, x, x == nx - 1 ? 0 : x + 1};
            float d[3] = {0.f, 0.f, 0.f};
            if (p.eq_mode == 0) {
                d[0] = (qx[t - x + xo[2]] - qx[t - x + xo[0]]) * p.inv_2lam[0];
                d[1] = (qy[2 * nx + t] - qy[t]) * p.inv_2lam[1];
            }
            T* const row[3] = {y == 0 ? dst_below : dst + t - x - nx, dst + t - x,
                               y == rows - 1 ? dst_above : dst + t - x + nx};
            auto put = [&](int i, float gn) {
                row[cy_of(i) + 1][i * plane + xo[cx_of(i) + 1]] = S::cvt(S::shifted ? gn : fmaf(p.bw[i], p.rho_ref, gn));
            };
            relax_streamed<2>(p, [&](int i) { return g[i]; }, put, drho, j, d, inv);
        };
        if (threadIdx.x < nodes) relax_node(threadIdx.x, g0, drho0, j0, inv0);
        for (int t = threadIdx.x + kClThreads; t < nodes; t += kClThreads) {
            float g[9], drho, j[3], inv;
            load(t, g, drho, j, inv);
            relax_node(t, g, drho, j, inv);
        }
        cur ^= 1;
        cluster.sync();  // the pushes have landed, the anomaly may be overwritten
    }
    const T* last = pops + cur * 9 * plane;
    for (int t = threadIdx.x; t < nodes; t += kClThreads)
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i * p.N + row0 * nx + t] = last[i * plane + t];
}

// Rows per block and shared memory of a block.
inline int cluster_band(const Solver& s) { return (s.ny + kClBlocks - 1) / kClBlocks; }
inline size_t cluster_smem(const Solver& s)
{
    const size_t band = cluster_band(s);
    return ((2 * band + 2) * 4 + 18 * band * storage_bytes(s.storage)) * s.nx;
}

// Grids the cluster takes: at most kClMaxNodes nodes a block.  us per step, cluster against
// march: 64 x 64 1.6 / 4.1, 96 x 96 (1152 nodes a block) 2.95 / 4.1 FP32 and 2.75 / 4.3
// FP16, 192 x 64 (1536) 3.35 / 4.1 and 3.15 / 4.35, 128 x 128 (2048) 4.4 / 4.2 and 3.9 / 4.4,
// 160 x 100 (2080) 4.3 / 4.2.
constexpr int kClMaxNodes = 3 * kClThreads;
// ... whose shared memory is largest in FP32 with one row of them a block (cluster_smem()).
constexpr size_t kClMaxSmem = (size_t)kClMaxNodes * (4 * 4 + 18 * 4);
static_assert(kClMaxSmem <= 227 * 1024, "a band must fit the shared memory of a block");

// Launch configuration of the cluster of s.
struct ClusterLaunch {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    explicit ClusterLaunch(const Solver& s)
    {
        const int band = cluster_band(s);
        cfg.gridDim = dim3((unsigned)((s.ny + band - 1) / band));
        cfg.blockDim = dim3(kClThreads);
        cfg.dynamicSmemBytes = cluster_smem(s);
        cfg.stream = s.stream;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = cfg.gridDim.x;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
};

// Whether the device can hold the cluster (asked once per solver).
template <int ST>
bool cluster_fits(const Solver& s)
{
    if (s.cluster_ok < 0) {
        int clusters = 0;
        ClusterLaunch l(s);
        cudaError_t e = set_smem_limit_once<k_cluster_d2q9<ST>>((int)kClMaxSmem);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&clusters, k_cluster_d2q9<ST>, &l.cfg);
        if (e != cudaSuccess) (void)cudaGetLastError();
        s.cluster_ok = e == cudaSuccess && clusters > 0 ? 1 : 0;
    }
    return s.cluster_ok == 1;
}

// Steps of a call from which the cluster is the faster one: loading and storing the
// grid costs as much as one to four steps of the march, more where three rows leave it
// three blocks, less where the march's blocks do not find an SM each.  us a call, cluster
// against march, FP32 (FP16): 64 x 64, one node a thread, 2 steps 8.2 / 8.0 (6.4 / 8.2);
// 512 x 3 2 steps 8.2 / 7.2, 3 steps 10.3 / 10.8; 128 x 64, two nodes, 3 steps 12.3 / 12.3,
// 5 steps 17.6 / 20.5; 192 x 64, three nodes, 5 steps 22.6 / 20.5 (20.5 / 21.8), 50 steps 168 /
// 205; 1536 x 3 5 steps 22.6 / 18.4, 50 steps 174 / 183; 12 x 1000, 250 blocks of the march,
// 2 steps 12.3 / 13.1.
inline int cluster_min_steps(const Solver& s)
{
    const int nodes = cluster_band(s) * s.nx, seg = d2q9_segment_rows(s);
    const int march_blocks = (s.nx + kD2Cols - 1) / kD2Cols * ((s.ny + seg - 1) / seg);
    const bool many_rows = s.ny >= kClBlocks;
    if (march_blocks > s.num_sms || (nodes <= kClThreads && many_rows)) return 2;
    return nodes <= kClThreads ? 3 : nodes <= 2 * kClThreads ? 5 : many_rows ? 8 : 16;
}

// Whether a call of nsteps steps of s takes the cluster.
inline bool cluster_d2q9_applies(const Solver& s, int nsteps)
{
    if (s.D != 2 || (long long)cluster_band(s) * s.nx > kClMaxNodes) return false;
    if (nsteps < cluster_min_steps(s)) return false;
    switch (s.storage) {
        case ELBM_F32: return cluster_fits<ELBM_F32>(s);
        case ELBM_F32_SHIFT: return cluster_fits<ELBM_F32_SHIFT>(s);
        case ELBM_F16_SHIFT: return cluster_fits<ELBM_F16_SHIFT>(s);
        default: return cluster_fits<ELBM_BF16_SHIFT>(s);
    }
}

inline cudaError_t steps_cluster_d2q9(const Solver& s, int nsteps, long long* launches)
{
    StepParams p;
    fill_params(s, p);
    p.parity = 0;
    const ClusterLaunch l(s);
    cudaError_t e = cudaSuccess;
    for (int left = nsteps; left > 0 && e == cudaSuccess; left -= kClMaxSteps) {
        ELBM_DISPATCH_STORAGE(s.storage, {
            e = cudaLaunchKernelEx(&l.cfg, k_cluster_d2q9<ST>, p, cluster_band(s), std::min(left, kClMaxSteps));
        });
        if (e == cudaSuccess) ++*launches;
    }
    return e;
}

}  // namespace elbm
