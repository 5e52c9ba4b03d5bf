// The TMEM single pass on any periodic D3Q27 grid: tile_x x tile_y tiles that may
// stick out of the grid, loaded by cp.async (tmem_tile_step with PB != 0).  Taken
// where the TMA-fed kernels do not apply.
//
// Bound as the TMA-fed kernel is, plus the idle nodes of tiles that stick out.  us per
// step, one launch per step of the cp.async-staged kernel with block-wide barriers that it
// replaces against this one: 180 x 120 x 100 FP32-shift 223 / 108, FP16 (rows on 8 bytes)
// 179 / 122; 161^3 507 / 313 and 416 / 271; 33 x 200 x 100 98 / 70 and 84 / 66; 3^3 15.4 /
// 8.4.  (With a loop per row in the copies and the ring rows all on one warp, the copies'
// latency bounded the 4-byte forms: 161^3 750 and 662, 33 x 200 x 100 192 and 167.)
#include "single_pass_tmem.cuh"

namespace elbm {

namespace {

template <int ST, int TX, int NT, int PB>
__global__ void __launch_bounds__(kTmThreads, 1)
    k_single_pass_ragged(const __grid_constant__ StepParams p, void* dst, int seg)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int z0 = blockIdx.z * seg;
    tmem_tile_step<ST, TX, NT, false, false, PB>(nullptr, nullptr, p, dst, blockIdx.x * TX,
                                                 blockIdx.y * (kTmConsumers / TX), z0, min(p.nz, z0 + seg), smem_raw);
}

template <int ST, int TX, int PB>
cudaError_t launch(const Solver& s, const StepParams& p, void* dst)
{
    constexpr int TY = kTmConsumers / TX, NT = sizeof(typename Storage<ST>::T) == 4 && TX == 32 ? 1 : 2;
    const int smem = TmemLayout<ST, TX, NT, PB>::bytes;
    cudaError_t e = set_smem_limit_once<k_single_pass_ragged<ST, TX, NT, PB>>(smem);
    if (e != cudaSuccess) return e;
    const int seg = solver_segment_planes(s, TX, TY, 1);
    const dim3 grid((unsigned)((s.nx + TX - 1) / TX), (unsigned)((s.ny + TY - 1) / TY), (unsigned)((s.nz + seg - 1) / seg));
    return launch_pdl(k_single_pass_ragged<ST, TX, NT, PB>, grid, dim3(kTmThreads), smem, s.stream, p, dst, seg);
}

}  // namespace

// Tiles of 64 x 8 or 32 x 16 columns, whichever cover the grid with fewer nodes
// (64-wide ones when equal, see launch_single_tmem()); 16-byte pieces where rows
// start on 16 bytes, else 4-byte words.
cudaError_t launch_single_ragged(const Solver& s, const StepParams& p, void* dst)
{
    auto covered = [&](long long tx, long long ty) { return (s.nx + tx - 1) / tx * tx * ((s.ny + ty - 1) / ty * ty); };
    const bool wide = covered(64, 8) <= covered(32, 16);
    const bool aligned = (s.nx * storage_bytes(s.storage)) % 16 == 0 && (uintptr_t)p.f % 16 == 0;
    ELBM_DISPATCH_STORAGE(s.storage, {
        if (aligned) return wide ? launch<ST, 64, 16>(s, p, dst) : launch<ST, 32, 16>(s, p, dst);
        return wide ? launch<ST, 64, 4>(s, p, dst) : launch<ST, 32, 4>(s, p, dst);
    });
    return cudaErrorInvalidValue;
}

}  // namespace elbm
