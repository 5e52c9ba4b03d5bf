// The in-place two-pass step with walls and body force (the turbulent channel
// setup of Sec. III.E): half-way bounce-back below y = 0 and above y = ny-1,
// the anomaly's ghost value beyond a wall in the central difference of
// Eq. Paastar1, and the exact-difference body-force increment.  The same
// kernels as the periodic step, instantiated with BC = true, which reads the
// wall and force switches from the parameter block; kept in their own
// translation units so that the periodic kernels compile without them.
#pragma once
#include "step_kernels.cuh"

namespace elbm {

template <int D, int ST, int PAR, bool FX>
void launch_bounded(const StepParams& p, dim3 grid, cudaStream_t st, long long* launches)
{
    if (p.eq_mode == 2) {
        k_collide<D, ST, PAR, true, true, FX><<<grid, kBlock, 0, st>>>(p);
    } else {
        if (p.eq_mode == 0) {
            k_anomaly<D, ST, PAR, true><<<grid, kBlock, 0, st>>>(p);
            ++*launches;
        }
        k_collide<D, ST, PAR, false, true, FX><<<grid, kBlock, 0, st>>>(p);
    }
    ++*launches;
}

// A force along x alone (or none) takes the lighter force increment, whose registers
// let the collide kernel gather into registers (collide_in_registers()).
template <int D>
cudaError_t step_bounded_impl(const Solver& s, int parity, long long* launches)
{
    StepParams p;
    fill_params(s, p);
    p.parity = parity;
    const dim3 grid((unsigned)((s.N + kBlock - 1) / kBlock));
    const bool fx = p.g[1] == 0.f && p.g[2] == 0.f;
    ELBM_DISPATCH_STORAGE(s.storage, {
        if (parity == 0)
            fx ? launch_bounded<D, ST, 0, true>(p, grid, s.stream, launches)
               : launch_bounded<D, ST, 0, false>(p, grid, s.stream, launches);
        else
            fx ? launch_bounded<D, ST, 1, true>(p, grid, s.stream, launches)
               : launch_bounded<D, ST, 1, false>(p, grid, s.stream, launches);
    });
    return cudaGetLastError();
}

}  // namespace elbm
