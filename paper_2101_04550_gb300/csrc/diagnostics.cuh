// FP64 diagnostics of the current state: the reductions of elbm_reduce, the
// Fourier-mode projection of elbm_mode_sums and the field sums of the automatic
// storage baseline.
#pragma once
#include <cfloat>

#include "single_pass.cuh"

namespace elbm {

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_min(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ double warp_max(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ double red_combine(int k, double a, double b)
{
    return k == 9 ? fmin(a, b) : k == 11 ? fmax(a, b) : a + b;
}
__device__ __forceinline__ double red_warp(int k, double v)
{
    return k == 9 ? warp_min(v) : k == 11 ? warp_max(v) : warp_sum(v);
}

// Reduce the first NQ of ELBM_NRED FP64 accumulators over the block (kBlock threads):
// warp shuffles, then one shared-memory stage.
template <int NQ>
__device__ __forceinline__ void block_reduce(const double* acc, double* out)
{
    __shared__ double sh[kBlock / 32][NQ];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NQ; ++k) {
        const double v = red_warp(k, acc[k]);
        if (lane == 0) sh[warp][k] = v;
    }
    __syncthreads();
    if (threadIdx.x < NQ) {
        const int k = threadIdx.x;
        double v = sh[0][k];
        for (int w = 1; w < kBlock / 32; ++w) v = red_combine(k, v, sh[w][k]);
        out[k] = v;
    }
}

// Last stage of a reduction kernel, taken by the block that finishes last: fold the
// partials of `rows` blocks in a fixed order (deterministic), a warp per quantity,
// and put the solver's status word behind the ELBM_NRED results, so that one copy
// brings both to the host.  `partials` are this kernel's own (already written by
// every block) and, before them, those of earlier kernels on the stream; *counter is
// zero between launches.  (A kernel of its own for this took 14 us and a launch.)
__device__ __forceinline__ void finish_reduction(const double* partials, int rows, int nq, unsigned* counter,
                                                 const int* status, double* out)
{
    __shared__ bool last;
    __threadfence();  // this block's partials, before it counts itself done
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int lane = threadIdx.x & 31;
    for (int k = threadIdx.x >> 5; k < nq; k += kBlock / 32) {
        auto fold = [&](double none, auto&& op) {
            constexpr int U = 8;  // independent chains, and loads in flight
            double v[U];
#pragma unroll
            for (int j = 0; j < U; ++j) v[j] = none;
            for (int b0 = lane; b0 < rows; b0 += 32 * U)
#pragma unroll
                for (int j = 0; j < U; ++j)
                    if (b0 + 32 * j < rows) v[j] = op(v[j], __ldcg(partials + (size_t)(b0 + 32 * j) * ELBM_NRED + k));
#pragma unroll
            for (int w = U / 2; w > 0; w /= 2)
#pragma unroll
                for (int j = 0; j < w; ++j) v[j] = op(v[j], v[j + w]);
            return v[0];
        };
        double v;
        if (k == 9) v = warp_min(fold(DBL_MAX, [](double a, double b) { return fmin(a, b); }));
        else if (k == 11) v = warp_max(fold(0.0, [](double a, double b) { return fmax(a, b); }));
        else v = warp_sum(fold(0.0, [](double a, double b) { return a + b; }));
        if (lane == 0) out[k] = v;
    }
    if (threadIdx.x == 0) {
        out[ELBM_NRED] = (double)*status;
        *counter = 0;
    }
}

// Compensated FP32 sum: each addition is split exactly into its rounded sum and the
// rounding error (Knuth's TwoSum), and the errors accumulate in lo.  lo grows by up to
// half a unit in the last place of hi a term, and with it the rounding of lo itself, so
// a thread folds lo back into hi (Dekker's FastTwoSum) every kFold terms: hi + lo is
// then within about kFold n 2^-49 of the exact sum relative to the sum of the terms'
// magnitudes, for any number of terms n (up to 700 of D3Q27, 2000 of D2Q9 a thread).
// Without the fold it is n^2 2^-50: a thread's 0.1 followed by 574 terms of 3e-9 came out
// 6e-11 off.  Per-thread partial sums so keep FP64-grade accuracy while the arithmetic
// stays on the FP32 pipes (FP64 issue is far slower on this GPU); the sums across threads
// and blocks are FP64.  Folding costs the reductions of an FP32 grid 0.5 % at 256^3, 2.5 % at
// 135 x 121 x 150 and 5 % at 4096^2, however often.
struct Sum2f {
    static constexpr int kFold = 8;
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float x)
    {
        const float s = hi + x;
        const float bp = s - hi;
        const float err = (hi - (s - bp)) + (x - bp);
        hi = s;
        lo += err;
    }
    __device__ __forceinline__ void fold()
    {
        const float s = hi + lo;
        lo -= s - hi;
        hi = s;
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// ----------------------------------------------------------- elbm_reduce
// Two kernels.  k_red_nodes reads the populations once, forms rho, u and min f of
// every node (FP32, the step kernels' sums), adds the terms that need no
// neighbour and writes u to scratch vel[D][N]; k_red_gradients adds the terms of
// vorticity and d_x u_x by central differences of vel (node spacing lam) and the
// wall-normal gradient.  Partials are FP64 per block, compensated FP32 within a
// thread.
//
// Bound by HBM: reading 108 B and writing 12 B per FP32 node, 296 us at 256^3, then
// reading 12 B, 30 us; 317 + 90 us are measured (297 + 222 us when the
// sums all sat in the second kernel and rho and min f went through scratch too).
// One kernel that marches tiles with a ring of recomputed nodes needs no scratch
// but 450 instructions a node and took 468 us (754 us with its populations staged
// by 4-byte cp.async).
template <int D, int ST>
__global__ void __launch_bounds__(kBlock, 3) k_red_nodes(const __grid_constant__ StepParams p, float* vel, double* partials)
{
    Sum2f mass, mom[3], rho_u2, u2, ux2;
    float fmin_ = FLT_MAX, umax = 0.f;
    int nonfinite = 0, terms = 0;
    for (int cell = blockIdx.x * kBlock + threadIdx.x; cell < p.N; cell += gridDim.x * kBlock) {
        const Node n = make_node<D>(p, cell);
        float g[Lat<D>::Q];
        gather_any<D, ST>(p, n, g);
        float drho, j[3], u[3] = {0.f, 0.f, 0.f};
        moments<D>(p, g, drho, j);
#pragma unroll
        for (int i = 0; i < Lat<D>::Q; ++i) fmin_ = fminf(fmin_, fmaf(p.bw[i], p.rho_ref, g[i]));
        const float r = p.rho_ref + drho;
        const float inv_r = 1.0f / r;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            u[a] = j[a] * inv_r + 0.5f * p.g[a];
            vel[(size_t)a * p.N + cell] = u[a];
            mom[a].add(r * u[a]);
        }
        const float uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
        const bool finite = isfinite(r) && isfinite(uu);
        mass.add(r);
        rho_u2.add(r * uu);
        u2.add(uu);
        ux2.add(u[0] * u[0]);
        nonfinite += finite ? 0 : 1;
        umax = fmaxf(umax, finite ? sqrtf(uu) : 0.f);
        if (++terms % Sum2f::kFold == 0) {
            mass.fold();
#pragma unroll
            for (int a = 0; a < D; ++a) mom[a].fold();
            rho_u2.fold();
            u2.fold();
            ux2.fold();
        }
    }
    double acc[ELBM_NRED] = {mass.value(),   mom[0].value(), mom[1].value(), mom[2].value(), rho_u2.value(), u2.value(),
                             0.0,            0.0,            ux2.value()};
    acc[9] = fmin_ == FLT_MAX ? DBL_MAX : (double)fmin_;
    acc[10] = (double)nonfinite;
    acc[11] = (double)umax;
    block_reduce<ELBM_NRED>(acc, partials + (size_t)blockIdx.x * ELBM_NRED);
}

// With walls the velocity beyond a wall is the negated value of the
// wall-adjacent node (no slip half-way between the nodes), and the wall-normal
// gradient of u_x at each wall node comes from the quadratic through the wall
// (u = 0, a distance lam_y/2 away) and the first two nodes:
// (9 u_x(1st) - u_x(2nd)) / (3 lam_y).
// V: nodes a thread takes at once along x (4 where rows are whole 16-byte pieces).
// A node needs 14 neighbour values, and the load unit bounds one load each
// (160 us at 256^3); four nodes share 11 16-byte loads and 6 words (90 us).
template <int D, int V>
__global__ void __launch_bounds__(kBlock) k_red_gradients(const __grid_constant__ StepParams p, const float* __restrict__ vel,
                                                          double* partials, int node_rows, unsigned* counter, double* out)
{
    Sum2f curl2, dxux2, wall;
    int terms = 0;
    const bool walls = p.walls_y != 0;
    const float* ux = vel;
    const float* uy = vel + p.N;
    const float* uz = vel + 2 * (size_t)p.N;
    const float ix = 0.5f / p.lam[0], iy = 0.5f / p.lam[1], iz = 0.5f / p.lam[2];
    struct Piece {
        float v[V];
    };
    auto piece = [](const float* f, int cell) {
        Piece q;
        if (V == 4) {
            const float4 w = *reinterpret_cast<const float4*>(f + cell);
            q.v[0] = w.x;
            q.v[V > 1 ? 1 : 0] = w.y;
            q.v[V > 2 ? 2 : 0] = w.z;
            q.v[V > 3 ? 3 : 0] = w.w;
        } else {
            q.v[0] = f[cell];
        }
        return q;
    };
    for (int cell = (blockIdx.x * kBlock + threadIdx.x) * V; cell < p.N; cell += gridDim.x * kBlock * V) {
        const Node n = make_node<D>(p, cell);
        const int row = n.oy[1] + n.oz[1], yp = n.at(0, 1, 0), ym = n.at(0, -1, 0);
        const int left = n.at(-1, 0, 0), right = row + (n.ox[1] + V == p.nx ? 0 : n.ox[1] + V);
        const Piece x = piece(ux, cell), y = piece(uy, cell), z = (D == 3) ? piece(uz, cell) : Piece{};
        auto dx = [&](const Piece& q, float l, float r, int k) {
            return ((k < V - 1 ? q.v[k < V - 1 ? k + 1 : 0] : r) - (k > 0 ? q.v[k > 0 ? k - 1 : 0] : l)) * ix;
        };
        const float xl = ux[left], xr = ux[right], yl = uy[left], yr = uy[right];
        const float zl = (D == 3) ? uz[left] : 0.f, zr = (D == 3) ? uz[right] : 0.f;
        const Piece xu = piece(ux, yp), xd = piece(ux, ym);
        const Piece zu = (D == 3) ? piece(uz, yp) : Piece{}, zd = (D == 3) ? piece(uz, ym) : Piece{};
        Piece xa{}, xb{}, ya{}, yb{};  // u_x, u_y of the planes above and below
        if (D == 3) {
            xa = piece(ux, n.at(0, 0, 1));
            xb = piece(ux, n.at(0, 0, -1));
            ya = piece(uy, n.at(0, 0, 1));
            yb = piece(uy, n.at(0, 0, -1));
        }
#pragma unroll
        for (int k = 0; k < V; ++k) {
            auto dy = [&](const Piece& v, const Piece& up, const Piece& dn) {
                return (((walls && n.yhi) ? -v.v[k] : up.v[k]) - ((walls && n.ylo) ? -v.v[k] : dn.v[k])) * iy;
            };
            const float dxux = dx(x, xl, xr, k), wz = dx(y, yl, yr, k) - dy(x, xu, xd);
            float w2 = wz * wz;
            if (D == 3) {
                const float wx = dy(z, zu, zd) - (ya.v[k] - yb.v[k]) * iz, wy = (xa.v[k] - xb.v[k]) * iz - dx(z, zl, zr, k);
                w2 += wx * wx + wy * wy;
            }
            if (walls && (n.ylo || n.yhi))
                wall.add((9.0f * x.v[k] - (n.ylo ? xu : xd).v[k]) * (1.0f / (3.0f * p.lam[1])));
            curl2.add(w2);
            dxux2.add(dxux * dxux);
        }
        if ((terms += V) % Sum2f::kFold == 0) {
            curl2.fold();
            dxux2.fold();
            wall.fold();
        }
    }
    double acc[ELBM_NRED] = {};
    acc[6] = curl2.value();
    acc[7] = dxux2.value();
    acc[9] = DBL_MAX;
    acc[12] = wall.value();
    block_reduce<ELBM_NRED>(acc, partials + (size_t)(node_rows + blockIdx.x) * ELBM_NRED);
    finish_reduction(partials, node_rows + gridDim.x, ELBM_NRED, counter, p.status, out);
}

template <int D>
cudaError_t reduce_impl(const Solver& s, long long* launches)
{
    StepParams p;
    fill_params(s, p);
    // as many blocks as the GPU holds: a thread then sums over all its nodes
    const int nodes = std::min(s.red_blocks, 3 * s.num_sms);
    ELBM_DISPATCH_STORAGE(s.storage, {
        k_red_nodes<D, ST><<<nodes, kBlock, 0, s.stream>>>(p, s.vel, s.partials);
    });
    const int grads = std::min(s.red_blocks, 4 * s.num_sms);
    if (s.nx % 4 == 0)
        k_red_gradients<D, 4><<<grads, kBlock, 0, s.stream>>>(p, s.vel, s.partials, nodes, s.red_counter, s.red_out);
    else
        k_red_gradients<D, 1><<<grads, kBlock, 0, s.stream>>>(p, s.vel, s.partials, nodes, s.red_counter, s.red_out);
    *launches += 2;
    return cudaGetLastError();
}

// ------------------------------------------------- automatic storage baseline
// Sums of rho and rho u_a of a caller field (FP64), for the automatic storage
// baseline velocity: out[0] = sum rho, out[1 + a] = sum rho u_a.
template <int D, typename TIn>
__global__ void __launch_bounds__(kBlock) k_field_sums(int N, const TIn* rho, const TIn* u, double* partials,
                                                       unsigned* counter, const int* status, double* out)
{
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int cell = blockIdx.x * kBlock + threadIdx.x; cell < N; cell += gridDim.x * kBlock) {
        const double r = (double)rho[cell];
        acc[0] += r;
#pragma unroll
        for (int a = 0; a < D; ++a) acc[1 + a] += r * (double)u[(size_t)a * N + cell];
    }
    block_reduce<4>(acc, partials + (size_t)blockIdx.x * ELBM_NRED);
    finish_reduction(partials, gridDim.x, 4, counter, status, out);
}

template <int D>
cudaError_t field_sums_impl(const Solver& s, const void* rho, const void* u, int dtype, long long* launches)
{
    if (dtype == ELBM_DTYPE_F64)
        k_field_sums<D, double><<<s.red_blocks, kBlock, 0, s.stream>>>((int)s.N, (const double*)rho,
                                                                      (const double*)u, s.partials, s.red_counter,
                                                                      s.status, s.red_out);
    else
        k_field_sums<D, float><<<s.red_blocks, kBlock, 0, s.stream>>>((int)s.N, (const float*)rho,
                                                                     (const float*)u, s.partials, s.red_counter,
                                                                     s.status, s.red_out);
    ++*launches;
    return cudaGetLastError();
}

// --------------------------------------------------------- elbm_mode_sums
// Shear-mode projection (the amplitude of the shear wave, Sec. III.A):
// out[0] = sum_x (u . dir) cos(k . x), out[1] = sum_x (u . dir) sin(k . x), in
// FP64, with x = (i lam_x, j lam_y, k lam_z) the node's physical position and
// u the reported velocity.
//
// exp(i k . x) is the product of one factor per axis, so nx + ny + nz sines and
// cosines (k_mode_factors) serve the whole grid.  A block takes 32 columns x 64
// rows of a plane at a time, a warp every eighth row: a thread sums
// (u . dir) exp(i k_y y) over its rows and multiplies the sum by the x and z
// factors once.  That leaves 8 FP64 operations a node, which the reading of the
// populations hides (HBM floor 267 us at 256^3 FP32: 322 us); a sine and
// cosine of every node's phase took 1305 us, bound by FP64 issue.
struct ModeArgs {
    double k[3], dir[3];
};
constexpr int kModeRows = 64;

template <int D>
__global__ void __launch_bounds__(kBlock) k_mode_factors(StepParams p, ModeArgs m, double2* factors)
{
    const int t = blockIdx.x * kBlock + threadIdx.x;
    if (t >= p.nx + p.ny + p.nz) return;
    const int a = t < p.nx ? 0 : t < p.nx + p.ny ? 1 : 2;
    const int node = a == 0 ? t : a == 1 ? t - p.nx : t - p.nx - p.ny;
    double sn, cs;
    sincos(a < D ? m.k[a] * node * (double)p.lam[a] : 0.0, &sn, &cs);
    factors[t] = make_double2(cs, sn);
}

// u . dir of a node, in FP64.
template <int D, int ST>
__device__ __forceinline__ double mode_velocity(const StepParams& p, const Node& n, const ModeArgs& m)
{
    float g[Lat<D>::Q];
    gather_any<D, ST>(p, n, g);
    float drho, j[3];
    moments<D>(p, g, drho, j);
    const float inv_r = 1.0f / (p.rho_ref + drho);
    double us = 0.0;
#pragma unroll
    for (int a = 0; a < D; ++a) us += (double)(j[a] * inv_r + 0.5f * p.g[a]) * m.dir[a];
    return us;
}
__device__ __forceinline__ double2 complex_mul(double2 a, double2 b)
{
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

template <int D, int ST>
__global__ void __launch_bounds__(kBlock, 4)
    k_mode_sums(const __grid_constant__ StepParams p, ModeArgs m, const double2* factors, int chunks, int ysegs, int items,
                double* partials, unsigned* counter, double* out)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double acc[2] = {0.0, 0.0};
    for (int item = blockIdx.x; item < items; item += gridDim.x) {
        const int x = (item % chunks) * 32 + lane, y0 = (item / chunks % ysegs) * kModeRows, z = item / chunks / ysegs;
        const int y1 = min(p.ny, y0 + kModeRows);
        if (x >= p.nx) continue;
        double re = 0.0, im = 0.0;
        for (int y = y0 + warp; y < y1; y += kBlock / 32) {
            const double us = mode_velocity<D, ST>(p, make_node_at<D>(p, x, y, z), m);
            const double2 fy = factors[p.nx + y];
            re = fma(us, fy.x, re);
            im = fma(us, fy.y, im);
        }
        const double2 f = complex_mul(factors[x], factors[p.nx + p.ny + z]);
        acc[0] += re * f.x - im * f.y;
        acc[1] += re * f.y + im * f.x;
    }
    block_reduce<2>(acc, partials + (size_t)blockIdx.x * ELBM_NRED);
    finish_reduction(partials, gridDim.x, 2, counter, p.status, out);
}

// The same for grids whose planes leave most of a block's columns and rows without a
// node: a thread takes nodes one by one, whichever they are, and multiplies the three
// factors of each (14 FP64 operations more a node: a call takes 540 us at 256^3, 354 by
// rows).  mode_sums_impl() chooses.
template <int D, int ST>
__global__ void __launch_bounds__(kBlock, 4)
    k_mode_sums_nodes(const __grid_constant__ StepParams p, ModeArgs m, const double2* factors, double* partials,
                      unsigned* counter, double* out)
{
    double acc[2] = {0.0, 0.0};
    for (int cell = blockIdx.x * kBlock + threadIdx.x; cell < p.N; cell += gridDim.x * kBlock) {
        const int z = (D == 3) ? fast_div(cell, p.div_plane_m, p.div_plane_s) : 0, r = cell - z * p.plane;
        const int y = fast_div(r, p.div_nx_m, p.div_nx_s), x = r - y * p.nx;
        const double us = mode_velocity<D, ST>(p, make_node_at<D>(p, x, y, z), m);
        const double2 f = complex_mul(complex_mul(factors[x], factors[p.nx + y]), factors[p.nx + p.ny + z]);
        acc[0] = fma(us, f.x, acc[0]);
        acc[1] = fma(us, f.y, acc[1]);
    }
    block_reduce<2>(acc, partials + (size_t)blockIdx.x * ELBM_NRED);
    finish_reduction(partials, gridDim.x, 2, counter, p.status, out);
}

template <int D>
cudaError_t mode_sums_impl(const Solver& s, const double* k, const double* dir, long long* launches)
{
    StepParams p;
    fill_params(s, p);
    ModeArgs m;
    for (int a = 0; a < 3; ++a) {
        m.k[a] = k[a];
        m.dir[a] = dir[a];
    }
    double2* factors = reinterpret_cast<double2*>(s.factors);
    const int nf = s.nx + s.ny + s.nz, chunks = (s.nx + 31) / 32, ysegs = (s.ny + kModeRows - 1) / kModeRows;
    const int items = chunks * ysegs * s.nz;
    // Node by node where under three in eight of the threads find a node in a plane's
    // columns and the rows of a block's warps.  us a call, rows against nodes (and a sine and
    // cosine a node before both), FP32: 3 x 3 x 30000 230 / 45 (79), 8 x 8 x 4096 73 / 45 (79),
    // 3 x 128 x 512 81 / 44 (70), 128 x 3 x 512 (3/8) 52 / 44 (70), 15 x 30000 (15/32) 53 / 55
    // (92), 33 x 4000 (1/2) 35 / 41 (59), 20 x 20000 (5/8) 44 / 51 (87).
    constexpr int kWarps = kBlock / 32;
    const bool narrow = 8ll * s.nx * s.ny < 3 * 32ll * chunks * ((s.ny + kWarps - 1) / kWarps * kWarps);
    k_mode_factors<D><<<(nf + kBlock - 1) / kBlock, kBlock, 0, s.stream>>>(p, m, factors);
    ELBM_DISPATCH_STORAGE(s.storage, {
        if (narrow)
            k_mode_sums_nodes<D, ST><<<s.red_blocks, kBlock, 0, s.stream>>>(p, m, factors, s.partials, s.red_counter,
                                                                            s.red_out);
        else
            k_mode_sums<D, ST><<<std::min(items, s.red_blocks), kBlock, 0, s.stream>>>(p, m, factors, chunks, ysegs, items,
                                                                                      s.partials, s.red_counter, s.red_out);
    });
    *launches += 2;
    return cudaGetLastError();
}

}  // namespace elbm
