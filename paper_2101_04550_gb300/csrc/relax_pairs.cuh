// Relaxation of one D3Q27 node with the paired FP32 instructions.
//
// The arithmetic is relax_streamed() of step_kernels.cuh, rounding for rounding:
// the populations with c_x = -1 and c_x = +1 of each (c_y, c_z) go through the same
// operations, so they are taken as a pair (add / sub / mul / fma on .f32x2, each
// half rounded as the scalar instruction rounds it); the populations with
// c_x = 0, the axis factors and the sums of the increments stay scalar.  Products
// feed only fused multiply-adds or further products here, so there is no
// product-and-sum that could be contracted.
//
// The node's populations come in pair order (pair_slot()): slots 2 L and 2 L + 1
// hold the populations c_x = -1 and +1 of line L = (c_y + 1) + 3 (c_z + 1), slots
// 18 + L the population c_x = 0, so that a pair sits in a register pair.
#pragma once
#include "step_kernels.cuh"

namespace elbm {

__host__ __device__ constexpr int pair_slot(int i) { return i % 3 == 1 ? 18 + i / 3 : 2 * (i / 3) + (i % 3) / 2; }

struct f32x2 {
    unsigned long long v;
    __device__ __forceinline__ f32x2() {}
    __device__ __forceinline__ f32x2(float lo, float hi) { asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi)); }
    __device__ __forceinline__ void split(float& lo, float& hi) const
    {
        asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
    }
};
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

// BC, FX, drho, j, d, put: as relax_streamed(); inv_rho = 1 / (rho_ref + drho); g: the
// populations in pair order.
template <bool BC, bool FX, typename P>
__device__ __forceinline__ void relax_pairs(const StepParams& p, const float* g, P&& put, float drho, const float* j,
                                            const float* d, float inv_rho)
{
    float u[3], pcorr[3], du[3], dP[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        u[a] = __fmul_rn(j[a], inv_rho);
        pcorr[a] = __fmul_rn(__fmul_rn(p.coef, inv_rho), d[a]);
    }
    baseline_args<3>(p, u, pcorr, du, dP);
    const float om = p.omega;
    const bool forced = BC && p.forced;
    typename std::conditional<FX, ForceIncrementX<3>, ForceIncrement<3>>::type frc;
    if (forced) frc.init(p, (p.rho_ref + drho) / om, u);
    // axis factors, as for_each_equilibrium() forms them
    float A[3][3], dl[3][3], dlx_r[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float s = __fmul_rn(dP[a], p.inv_lam2[a]);
        const float t = __fmul_rn(du[a], p.inv_lam[a]);
        dl[a][0] = __fmul_rn(0.5f, __fsub_rn(s, t));
        dl[a][1] = -s;
        dl[a][2] = __fmul_rn(0.5f, __fadd_rn(s, t));
#pragma unroll
        for (int c = 0; c < 3; ++c) A[a][c] = __fadd_rn(p.base[a][c], dl[a][c]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) dlx_r[c] = __fmul_rn(p.rho_ref, dl[0][c]);
    f32x2 Az[3], dz[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        Az[c] = f32x2(A[2][c], A[2][c]);
        dz[c] = f32x2(dl[2][c], dl[2][c]);
    }
    const f32x2 drho2(drho, drho), om2(om, om);

    float e0 = 0.f, ex = 0.f, ey = 0.f, ez = 0.f;
    float keep[7], kf[7];
#pragma unroll
    for (int cy = 0; cy < 3; ++cy) {
        float pxy[3], dxy[3], row[3];
#pragma unroll
        for (int cx = 0; cx < 3; ++cx) {
            pxy[cx] = __fmul_rn(A[0][cx], A[1][cy]);
            dxy[cx] = fmaf(dlx_r[cx], A[1][cy], __fmul_rn(p.base_xr[cx], dl[1][cy]));
        }
        const f32x2 pxy2(pxy[0], pxy[2]), dxy2(dxy[0], dxy[2]), bxy2(p.bxy_pm[cy].x, p.bxy_pm[cy].y);
        f32x2 inc[3];
        float mid[3];
#pragma unroll
        for (int cz = 0; cz < 3; ++cz) {
            const int L = cy + 3 * cz, i = 3 * L;
            const f32x2 g2(g[2 * L], g[2 * L + 1]);
            const f32x2 geq2 = fma2(drho2, mul2(pxy2, Az[cz]), fma2(dxy2, Az[cz], mul2(bxy2, dz[cz])));
            inc[cz] = sub2(geq2, g2);
            if (cy == 1 && cz == 1) {
                geq2.split(keep[1], keep[2]);
                if (forced) {
                    kf[1] = frc(i);
                    kf[2] = frc(i + 2);
                }
            } else {
                const f32x2 out = fma2(om2, forced ? add2(inc[cz], f32x2(frc(i), frc(i + 2))) : inc[cz], g2);
                float lo, hi;
                out.split(lo, hi);
                put(i, lo);
                put(i + 2, hi);
            }
            const float gm = g[18 + L];
            const float geq = fmaf(drho, __fmul_rn(pxy[1], A[2][cz]),
                                   fmaf(dxy[1], A[2][cz], __fmul_rn(p.bxy_r[1 + 3 * cy], dl[2][cz])));
            mid[cz] = __fsub_rn(geq, gm);
            const int k = corrected_slot<3>(i + 1);
            if (k >= 0) {
                keep[k] = geq;
                if (forced) kf[k] = frc(i + 1);
            } else {
                put(i + 1, fmaf(om, forced ? mid[cz] + frc(i + 1) : mid[cz], gm));
            }
        }
        // the increments' moments, in the order of relax_streamed()
        add2(add2(inc[0], inc[1]), inc[2]).split(row[0], row[2]);
        row[1] = (mid[0] + mid[1]) + mid[2];
        float zm, zp;
        sub2(inc[2], inc[0]).split(zm, zp);
        ez += zm;
        ez += mid[2] - mid[0];
        ez += zp;
        const float rs = (row[0] + row[1]) + row[2];
        ex += row[2] - row[0];
        e0 += rs;
        if (cy == 2) ey += rs;
        if (cy == 0) ey -= rs;
    }
    auto incr = [&](int k, float v) { return forced ? v + kf[k] : v; };
    auto relaxed = [&](int k, int i, float h) {
        const float gi = g[pair_slot(i)];
        return fmaf(om, incr(k, __fadd_rn(__fsub_rn(keep[k], gi), h)), gi);
    };
    const float hx = __fmul_rn(0.5f, ex), hy = __fmul_rn(0.5f, ey), hz = __fmul_rn(0.5f, ez);
    put(13, relaxed(0, 13, -e0));
    put(12, relaxed(1, 12, hx));
    put(14, relaxed(2, 14, -hx));
    put(10, relaxed(3, 10, hy));
    put(16, relaxed(4, 16, -hy));
    put(4, relaxed(5, 4, hz));
    put(22, relaxed(6, 22, -hz));
}

}  // namespace elbm
