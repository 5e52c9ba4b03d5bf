// Kernels of the extended LBGK step and its utilities, templated on the
// lattice dimension D, the storage mode ST and (for the hot kernels) the AA
// streaming parity PAR.  Included by one translation unit per lattice.
#pragma once
#include <type_traits>

#include "lbm_device.cuh"

namespace elbm {

constexpr int kBlock = 256;

#define ELBM_DISPATCH_STORAGE(storage, ...)                              \
    switch (storage) {                                                   \
        case ELBM_F32: { constexpr int ST = ELBM_F32; __VA_ARGS__; } break;             \
        case ELBM_F32_SHIFT: { constexpr int ST = ELBM_F32_SHIFT; __VA_ARGS__; } break; \
        case ELBM_F16_SHIFT: { constexpr int ST = ELBM_F16_SHIFT; __VA_ARGS__; } break; \
        case ELBM_BF16_SHIFT: { constexpr int ST = ELBM_BF16_SHIFT; __VA_ARGS__; } break; \
        default: return cudaErrorInvalidValue;                           \
    }

// ---------------------------------------------------------------- two-pass
// Pass 1: post-streaming moments of every node -> anomaly field q[a][cell]
// (Eqs. density, momentum, Deviation).  Reads the populations only.  BC: the
// variant that honours walls (p.walls_y) and the body force (p.forced).
template <int D, int ST, int PAR, bool BC = false>
__global__ void __launch_bounds__(kBlock) k_anomaly(StepParams p)
{
    const int cell = blockIdx.x * kBlock + threadIdx.x;
    if (cell >= p.N) return;
    const Node n = make_node<D>(p, cell);
    float g[Lat<D>::Q];
    gather<D, ST, PAR>(p, n, g, BC && p.walls_y);
    float drho, j[3];
    moments<D>(p, g, drho, j);
    const float inv_rho = 1.0f / (p.rho_ref + drho);
#pragma unroll
    for (int a = 0; a < D; ++a) p.q[a * p.N + cell] = anomaly(p, a, j[a], j[a] * inv_rho);
}

// Moments of a node from a population accessor gval(i) (the sums of moments()).
template <int D, typename G>
__device__ __forceinline__ void moments_of(const StepParams& p, G&& gval, float& drho, float* j)
{
    // lines of three along x (population index x fastest), then rows along y, then planes along z
    constexpr int NL = Lat<D>::Q / 3, NP = NL / 3 > 0 ? NL / 3 : 1;
    float t[NL], sx = 0.f, sy = 0.f;
#pragma unroll
    for (int L = 0; L < NL; ++L) {
        const float a = gval(3 * L), b = gval(3 * L + 1), c = gval(3 * L + 2);
        t[L] = (a + b) + c;
        sx += c - a;
    }
    float tp[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int P = 0; P < NP; ++P) {
        tp[P] = (t[3 * P] + t[3 * P + 1]) + t[3 * P + 2];
        sy += t[3 * P + 2] - t[3 * P];
    }
    drho = (D == 3) ? (tp[0] + tp[1]) + tp[2] : tp[0];
    const float sz = (D == 3) ? tp[2] - tp[0] : 0.f;
    j[0] = fmaf(p.lam[0], sx, p.j0[0]);
    j[1] = fmaf(p.lam[1], sy, p.j0[1]);
    j[2] = (D == 3) ? fmaf(p.lam[2], sz, p.j0[2]) : 0.f;
}

// Relaxation of one node toward the extended equilibrium with the
// conservation correction of relax(), for populations read through gval(i)
// (read twice, not kept in registers) and results handed to put(i, g'_i).
// POLY selects the conventional second-order equilibrium instead.  BC adds
// the body-force increment F_i (ForceIncrement) when p.forced is set; it is
// kept out of the conservation moments, so the node gains exactly the
// momentum rho g of the force.  FX: the force is known to act along x alone
// (ForceIncrementX, same bits, fewer registers).  inv_rho, if given (> 0),
// is the caller's 1 / (rho_ref + drho), the very value computed here otherwise.
template <int D, bool POLY = false, bool BC = false, bool FX = false, typename G, typename P>
__device__ __forceinline__ void relax_streamed(const StepParams& p, G&& gval, P&& put, float drho,
                                               const float* j, const float* d, float inv_rho_in = 0.f)
{
    constexpr int I0 = (Lat<D>::Q - 1) / 2;
    const float rho = p.rho_ref + drho;
    const float inv_rho = inv_rho_in > 0.f ? inv_rho_in : 1.0f / rho;
    float u[3], pcorr[3], du[3], dP[3];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        u[a] = __fmul_rn(j[a], inv_rho);
        pcorr[a] = __fmul_rn(__fmul_rn(p.coef, inv_rho), d[a]);
    }
    baseline_args<D>(p, u, pcorr, du, dP);
    const float om = p.omega;
    const bool forced = BC && p.forced;
    typename std::conditional<FX, ForceIncrementX<D>, ForceIncrement<D>>::type frc;
    if (forced) frc.init(p, rho / om, u);
    float e0 = 0.f, ex = 0.f, ey = 0.f, ez = 0.f;
    float keep[2 * D + 1], kf[2 * D + 1];
    // the increments' moments, summed along the enumeration's lines: cz
    // innermost (D3Q27) or cx innermost (D2Q9), then cx, then cy
    float line[3], row[3];
    auto accumulate = [&](int i, float dl) {
        const int cx = cx_of(i), cy = cy_of(i);
        if (D == 3) {
            const int cz = cz_of<D>(i);
            line[cz + 1] = dl;
            if (cz != 1) return;
            row[cx + 1] = (line[0] + line[1]) + line[2];
            ez += line[2] - line[0];
        } else {
            row[cx + 1] = dl;
        }
        if (cx != 1) return;
        const float rs = (row[0] + row[1]) + row[2];
        ex += row[2] - row[0];
        e0 += rs;
        if (cy == 1) ey += rs;
        if (cy == -1) ey -= rs;
    };
    auto relax_one = [&](int i, float geq) {
        const float gi = gval(i);
        const float dl = __fsub_rn(geq, gi);
        accumulate(i, dl);
        const int k = corrected_slot<D>(i);
        if (k >= 0) {
            keep[k] = geq;
            if (forced) kf[k] = frc(i);
        } else {
            put(i, fmaf(om, forced ? dl + frc(i) : dl, gi));
        }
    };
    if (POLY) for_each_second_order<D>(p, drho, u, relax_one);
    else for_each_equilibrium<D>(p, drho, du, dP, relax_one);
    auto inc = [&](int k, float v) { return forced ? v + kf[k] : v; };
    const float hx = __fmul_rn(0.5f, ex), hy = __fmul_rn(0.5f, ey);
    // f*_k - f_k with the half-increment h of its axis: (keep - g) -+ h
    auto corr = [&](int k, int i, float h) { return inc(k, __fadd_rn(__fsub_rn(keep[k], gval(i)), h)); };
    put(I0, fmaf(om, inc(0, __fsub_rn(__fsub_rn(keep[0], gval(I0)), e0)), gval(I0)));
    put(I0 - 1, fmaf(om, corr(1, I0 - 1, hx), gval(I0 - 1)));
    put(I0 + 1, fmaf(om, corr(2, I0 + 1, -hx), gval(I0 + 1)));
    put(I0 - 3, fmaf(om, corr(3, I0 - 3, hy), gval(I0 - 3)));
    put(I0 + 3, fmaf(om, corr(4, I0 + 3, -hy), gval(I0 + 3)));
    if (D == 3) {
        const float hz = __fmul_rn(0.5f, ez);
        put(I0 - 9, fmaf(om, corr(5, I0 - 9, hz), gval(I0 - 9)));
        put(I0 + 9, fmaf(om, corr(6, I0 + 9, -hz), gval(I0 + 9)));
    }
}

// The per-node update once the anomaly field of this time level is complete:
// gather the post-streaming populations into the thread's shared-memory
// column `col` (stride STRIDE, the block size), central difference of q along each axis
// (Eq. Paastar1), extended equilibrium, relaxation, write-back in place.
// Populations are read back from the stage instead of being held in
// registers, which keeps the register count low enough for 32 resident
// warps per SM.  BC: walls (bounce-back slots, and the anomaly's ghost value
// beyond a wall is the negated value of the wall-adjacent node: Q~_yyy is odd
// in u_y and u_y = 0 on the wall) and the body force.
template <int D, int ST, int PAR, int STRIDE = kBlock, bool POLY = false, bool BC = false, bool FX = false>
__device__ __forceinline__ void collide_staged(const StepParams& p, int cell, unsigned* col)
{
    constexpr int Q = Lat<D>::Q;
    using S = Storage<ST>;
    const Node n = make_node<D>(p, cell);
    const bool walls = BC && p.walls_y;
    unsigned halves = 0;  // bit i: population i sits in the upper half of its staged word
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int idx = read_slot<D>(n, p.N, i, PAR, walls);
        halves |= (unsigned)(idx & 1) << i;
        cp_async4(col + i * STRIDE, stage_src<ST>(p, idx));
    }
    float d[3] = {0.f, 0.f, 0.f};
    if (p.eq_mode == 0) {
        const float* q = p.q;
        d[0] = (q[n.at(1, 0, 0)] - q[n.at(-1, 0, 0)]) * p.inv_2lam[0];
        const float* qy = q + p.N;
        const float qyp = (walls && n.yhi) ? -qy[cell] : qy[n.at(0, 1, 0)];
        const float qym = (walls && n.ylo) ? -qy[cell] : qy[n.at(0, -1, 0)];
        d[1] = (qyp - qym) * p.inv_2lam[1];
        if (D == 3) d[2] = (q[2 * p.N + n.at(0, 0, 1)] - q[2 * p.N + n.at(0, 0, -1)]) * p.inv_2lam[2];
    }
    cp_async_wait_all();
    auto gval = [&](int i) {
        const float v = stage_value<ST>(p, ld_stage(col + i * STRIDE), (int)((halves >> i) & 1u), i);
        return (S::shifted && PAR == 1 && walls && read_bounced(n, i)) ? v + bounce_rebase<D>(p, i) : v;
    };
    float drho, j[3];
    moments_of<D>(p, gval, drho, j);
    typename S::T* f = static_cast<typename S::T*>(p.f);
    const int cell_o = opaque(cell);
    auto put = [&](int i, float gn) {
        const int slot = (PAR == 0) ? (Q - 1 - i) * p.N + cell_o : write_slot<D>(n, p.N, i, PAR, walls);
        if (S::shifted && PAR == 1 && walls && write_bounced(n, i)) gn += bounce_rebase<D>(p, Q - 1 - i);
        S::store(f + slot, S::shifted ? gn : fmaf(p.bw[i], p.rho_ref, gn));
    };
    relax_streamed<D, POLY, BC, FX>(p, gval, put, drho, j, d);
}

// The same with the populations gathered into registers (27 loads in flight a thread,
// 24 warps an SM) instead of staged in shared memory by 4-byte cp.async (32 warps).
// Which one a kernel takes is collide_in_registers().
template <int D, int ST, int PAR, bool POLY = false, bool BC = false, bool FX = false>
__device__ __forceinline__ void collide_node(const StepParams& p, int cell)
{
    constexpr int Q = Lat<D>::Q;
    using S = Storage<ST>;
    const Node n = make_node<D>(p, cell);
    const bool walls = BC && p.walls_y;
    float g[Q];
    gather<D, ST, PAR>(p, n, g, walls);
    float d[3] = {0.f, 0.f, 0.f};
    if (p.eq_mode == 0) {
        const float* q = p.q;
        d[0] = (q[n.at(1, 0, 0)] - q[n.at(-1, 0, 0)]) * p.inv_2lam[0];
        const float* qy = q + p.N;
        const float qyp = (walls && n.yhi) ? -qy[cell] : qy[n.at(0, 1, 0)];
        const float qym = (walls && n.ylo) ? -qy[cell] : qy[n.at(0, -1, 0)];
        d[1] = (qyp - qym) * p.inv_2lam[1];
        if (D == 3) d[2] = (q[2 * p.N + n.at(0, 0, 1)] - q[2 * p.N + n.at(0, 0, -1)]) * p.inv_2lam[2];
    }
    auto gval = [&](int i) { return g[i]; };
    float drho, j[3];
    moments_of<D>(p, gval, drho, j);
    typename S::T* f = static_cast<typename S::T*>(p.f);
    const int cell_o = opaque(cell);
    auto put = [&](int i, float gn) {
        const int slot = (PAR == 0) ? (Q - 1 - i) * p.N + cell_o : write_slot<D>(n, p.N, i, PAR, walls);
        if (S::shifted && PAR == 1 && walls && write_bounced(n, i)) gn += bounce_rebase<D>(p, Q - 1 - i);
        S::store(f + slot, S::shifted ? gn : fmaf(p.bw[i], p.rho_ref, gn));
    };
    relax_streamed<D, POLY, BC, FX>(p, gval, put, drho, j, d);
}

// Where the register form is the faster one: 16-bit storage, D2Q9, unshifted FP32 and
// the periodic second-order equilibrium; not with the general body force, whose
// increment leaves no registers, nor for D3Q27 in 16 bits with the second-order
// equilibrium between walls, which spills.  us per two-pass step, registers against stage,
// 135 x 121 x 150: FP16 125 / 136, FP32 161 / 161, FP32-shift 167 / 158; walls and x force
// FP16 209 / 217, FP32 165 / 178, FP32-shift 200 / 190; second order FP16 76 / 93, FP32-shift
// 93 / 102; second order, walls and x force FP32 99 / 110, FP16 126 / 118, BF16 126 / 121,
// FP32-shift 136 / 125; D2Q9 2048^2 FP32 95 / 102, with those options FP32 61 / 65, FP16
// 50 / 62.
template <int D, int ST, bool POLY, bool BC, bool FX>
__host__ __device__ constexpr bool collide_in_registers()
{
    if (BC && !FX) return false;
    if (D == 3 && POLY && BC && sizeof(typename Storage<ST>::T) == 2) return false;
    return D == 2 || sizeof(typename Storage<ST>::T) == 2 || ST == ELBM_F32 || (POLY && !BC);
}
template <int D, int ST, bool POLY = false, bool BC = false, bool FX = false>
__host__ __device__ constexpr int collide_min_blocks()
{
    return collide_in_registers<D, ST, POLY, BC, FX>() || BC ? 3 : 4;
}

// Pass 2 over every node, one node per thread.  POLY: the conventional second-order
// equilibrium (no anomaly pass).  BC: walls and body force; FX: the force acts along
// x alone.
template <int D, int ST, int PAR, bool POLY = false, bool BC = false, bool FX = false>
__global__ void __launch_bounds__(kBlock, collide_min_blocks<D, ST, POLY, BC, FX>()) k_collide(StepParams p)
{
    const int cell = blockIdx.x * kBlock + threadIdx.x;
    if constexpr (collide_in_registers<D, ST, POLY, BC, FX>()) {
        if (cell < p.N) collide_node<D, ST, PAR, POLY, BC, FX>(p, cell);
    } else {
        __shared__ unsigned stage[Lat<D>::Q * kBlock];
        if (cell < p.N) collide_staged<D, ST, PAR, kBlock, POLY, BC, FX>(p, cell, stage + threadIdx.x);
    }
}

template <int D>
cudaError_t step_two_pass_impl(const Solver& s, int parity, long long* launches)
{
    StepParams p;
    fill_params(s, p);
    p.parity = parity;
    // walls and body force: the kernels of bounded_step.cuh (own translation units)
    if (p.walls_y || p.forced) return step_bounded_impl<D>(s, parity, launches);
    const dim3 grid((unsigned)((s.N + kBlock - 1) / kBlock));
    ELBM_DISPATCH_STORAGE(s.storage, {
        if (p.eq_mode == 2) {
            if (parity == 0) k_collide<D, ST, 0, true><<<grid, kBlock, 0, s.stream>>>(p);
            else k_collide<D, ST, 1, true><<<grid, kBlock, 0, s.stream>>>(p);
        } else if (parity == 0) {
            if (p.eq_mode == 0) { k_anomaly<D, ST, 0><<<grid, kBlock, 0, s.stream>>>(p); ++*launches; }
            k_collide<D, ST, 0><<<grid, kBlock, 0, s.stream>>>(p);
        } else {
            if (p.eq_mode == 0) { k_anomaly<D, ST, 1><<<grid, kBlock, 0, s.stream>>>(p); ++*launches; }
            k_collide<D, ST, 1><<<grid, kBlock, 0, s.stream>>>(p);
        }
        ++*launches;
    });
    return cudaGetLastError();
}

// -------------------------------------------------------------------- init
// f_i = rho Psi_i(u, T + u^2, lam) (Eq. 27eq) at every node, written to the
// even-parity slots.
template <int D, int ST, typename TIn>
__global__ void __launch_bounds__(kBlock) k_init(StepParams p, const TIn* rho, const TIn* u)
{
    using S = Storage<ST>;
    const int cell = blockIdx.x * kBlock + threadIdx.x;
    if (cell >= p.N) return;
    const float drho = (float)((double)rho[cell] - (double)p.rho_ref);
    float uu[3], zero[3] = {0.f, 0.f, 0.f}, du[3], dP[3];
#pragma unroll
    for (int a = 0; a < D; ++a) uu[a] = (float)u[(size_t)a * p.N + cell];
    baseline_args<D>(p, uu, zero, du, dP);
    typename S::T* f = static_cast<typename S::T*>(p.f);
    for_each_equilibrium<D>(p, drho, du, dP, [&](int i, float geq) {
        S::store(f + i * p.N + cell, S::shifted ? geq : geq + p.bw[i] * p.rho_ref);
    });
}

template <int D>
cudaError_t init_impl(const Solver& s, const void* rho, const void* u, int dtype, long long* launches)
{
    StepParams p;
    fill_params(s, p);
    const dim3 grid((unsigned)((s.N + kBlock - 1) / kBlock));
    ELBM_DISPATCH_STORAGE(s.storage, {
        if (dtype == ELBM_DTYPE_F64)
            k_init<D, ST, double><<<grid, kBlock, 0, s.stream>>>(p, (const double*)rho, (const double*)u);
        else
            k_init<D, ST, float><<<grid, kBlock, 0, s.stream>>>(p, (const float*)rho, (const float*)u);
        ++*launches;
    });
    return cudaGetLastError();
}

// ------------------------------------------------------------- read-outs
// Post-streaming populations of a node as deviations g_i, at the solver's
// current parity (not a hot path: parity is a run-time value here).  Shifted storage
// without walls has a branch of its own: the test for a bounced slot behind every load
// kept the loads from being in flight together (at odd parity elbm_reduce 256^3 FP16
// 882 us, 519 before its sums moved to the node pass, now 437; FP32-shift 613, 453;
// the mode projection 636, 354 and 581, 382).  Unshifted FP32 has nothing to rebase.
template <int D, int ST>
__device__ __forceinline__ void gather_any(const StepParams& p, const Node& n, float* g)
{
    constexpr bool rebase = Storage<ST>::shifted;
    if (p.parity == 0) gather<D, ST, 0>(p, n, g);
    else if (rebase && !p.walls_y) gather<D, ST, 1>(p, n, g);
    else gather<D, ST, 1>(p, n, g, rebase || p.walls_y != 0);
}

// rho and u of every node (Eqs. density, momentum) with the step kernels'
// FP32 sums; with a body force u is reported at the half step, u + g/2.
template <int D, int ST, typename TOut>
__global__ void __launch_bounds__(kBlock) k_moments(StepParams p, TOut* rho, TOut* u)
{
    const int cell = blockIdx.x * kBlock + threadIdx.x;
    if (cell >= p.N) return;
    const Node n = make_node<D>(p, cell);
    float g[Lat<D>::Q];
    gather_any<D, ST>(p, n, g);
    float drho, j[3];
    moments<D>(p, g, drho, j);
    const float r = p.rho_ref + drho;
    const float inv_r = 1.0f / r;
    rho[cell] = (TOut)r;
#pragma unroll
    for (int a = 0; a < D; ++a) u[(size_t)a * p.N + cell] = (TOut)(j[a] * inv_r + 0.5f * p.g[a]);
}

template <int D>
cudaError_t moments_impl(const Solver& s, void* rho, void* u, int dtype, long long* launches)
{
    StepParams p;
    fill_params(s, p);
    const dim3 grid((unsigned)((s.N + kBlock - 1) / kBlock));
    ELBM_DISPATCH_STORAGE(s.storage, {
        if (dtype == ELBM_DTYPE_F64)
            k_moments<D, ST, double><<<grid, kBlock, 0, s.stream>>>(p, (double*)rho, (double*)u);
        else
            k_moments<D, ST, float><<<grid, kBlock, 0, s.stream>>>(p, (float*)rho, (float*)u);
        ++*launches;
    });
    return cudaGetLastError();
}

// Post-streaming population i of a node, unshifted, in FP32 or FP64.
template <int D, int ST, typename TOut>
__device__ __forceinline__ TOut load_unshifted(const StepParams& p, const Node& n, int i)
{
    using S = Storage<ST>;
    const typename S::T* f = static_cast<const typename S::T*>(p.f);
    const bool walls = p.walls_y != 0;
    const float v = S::load(f + read_slot<D>(n, p.N, i, p.parity, walls));
    // a bounced slot holds population opp(i), stored against its own baseline
    const int b = (p.parity == 1 && walls && read_bounced(n, i)) ? Lat<D>::Q - 1 - i : i;
    if (!S::shifted) return (TOut)v;
    if (sizeof(TOut) == 4) return (TOut)fmaf(p.bw[b], p.rho_ref, v);
    return (TOut)((double)v + (double)p.bw[b] * (double)p.rho_ref);
}

// Unshifted post-streaming populations f_i = g_i + w_i rho_ref, layout f[i][cell].
// FP32 output of the read-out (and FP32 input of k_set_f below) takes one fused
// multiply-add instead of an FP64 sum rounded to FP32.  Bound by HBM: 27 loads
// and 27 stores a node, all loads in flight before the first store (FP32 storage
// and fields, 135 x 121 x 150: 77 us, floor 78; load and store by turns, as
// the compiler must order them when the arrays may alias, took 128).
template <int D, int ST, typename TOut>
__global__ void __launch_bounds__(kBlock) k_get_f(StepParams p, TOut* out)
{
    const int cell = blockIdx.x * kBlock + threadIdx.x;
    if (cell >= p.N) return;
    const Node n = make_node<D>(p, cell);
    TOut v[Lat<D>::Q];  // every load before the first store, which might alias
#pragma unroll
    for (int i = 0; i < Lat<D>::Q; ++i) v[i] = load_unshifted<D, ST, TOut>(p, n, i);
#pragma unroll
    for (int i = 0; i < Lat<D>::Q; ++i) out[(size_t)i * p.N + cell] = v[i];
}

// Store caller populations at the even-parity slots.
template <int D, int ST, typename TIn>
__global__ void __launch_bounds__(kBlock) k_set_f(StepParams p, const TIn* in)
{
    using S = Storage<ST>;
    const int cell = blockIdx.x * kBlock + threadIdx.x;
    if (cell >= p.N) return;
    typename S::T* f = static_cast<typename S::T*>(p.f);
    TIn v[Lat<D>::Q];
#pragma unroll
    for (int i = 0; i < Lat<D>::Q; ++i) v[i] = in[(size_t)i * p.N + cell];
#pragma unroll
    for (int i = 0; i < Lat<D>::Q; ++i) {
        float stored = (float)v[i];
        if (S::shifted)
            stored = sizeof(TIn) == 4 ? fmaf(-p.bw[i], p.rho_ref, (float)v[i])
                                      : (float)((double)v[i] - (double)p.bw[i] * (double)p.rho_ref);
        S::store(f + i * p.N + cell, stored);
    }
}

template <int D>
cudaError_t get_populations_impl(const Solver& s, void* f, int dtype, long long* launches)
{
    StepParams p;
    fill_params(s, p);
    const dim3 grid((unsigned)((s.N + kBlock - 1) / kBlock));
    ELBM_DISPATCH_STORAGE(s.storage, {
        if (dtype == ELBM_DTYPE_F64) k_get_f<D, ST, double><<<grid, kBlock, 0, s.stream>>>(p, (double*)f);
        else k_get_f<D, ST, float><<<grid, kBlock, 0, s.stream>>>(p, (float*)f);
        ++*launches;
    });
    return cudaGetLastError();
}

template <int D>
cudaError_t set_populations_impl(const Solver& s, const void* f, int dtype, long long* launches)
{
    StepParams p;
    fill_params(s, p);
    const dim3 grid((unsigned)((s.N + kBlock - 1) / kBlock));
    ELBM_DISPATCH_STORAGE(s.storage, {
        if (dtype == ELBM_DTYPE_F64) k_set_f<D, ST, double><<<grid, kBlock, 0, s.stream>>>(p, (const double*)f);
        else k_set_f<D, ST, float><<<grid, kBlock, 0, s.stream>>>(p, (const float*)f);
        ++*launches;
    });
    return cudaGetLastError();
}

}  // namespace elbm
