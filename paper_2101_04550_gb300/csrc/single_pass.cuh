// Single-pass form of the extended LBGK step with two population arrays: what its
// kernels share (segment depth, dependent launch, periodic index helpers).
//
// The correction term needs the anomaly Q~_aaa of the face neighbours at the
// same time level (Eq. Paastar1).  With a read-only source array and a
// separate destination, every block can recompute the anomaly of the nodes
// around its own tile, so one pass and one read of the populations suffice.
//
// State: `src` holds the post-streaming populations of every node at the
// node's own location (the layout of the in-place form's even parity).  A step
// reads src[i][x], relaxes, and pushes f'_i(x) to dst[i][x + c_i] (Eq. LBGK);
// then the arrays swap roles.
#pragma once
#include <algorithm>
#include <atomic>
#include <utility>
#include "step_kernels.cuh"

namespace elbm {

constexpr int kTileX = 32, kTileY = 8;   // kTileX * kTileY == kBlock

// Planes per segment of a D3Q27 single-pass launch.  A block marches through
// one tile column's segment of z planes and reads two planes more than it
// relaxes, so long segments re-read little and short ones fill the GPU.  The
// depth (up to 64) is the one whose schedule ends first when the blocks, in
// launch order, take the next free of `slots` resident places and a segment
// of n planes costs n + 2.5: a march is a serial chain of planes plus the block's
// start-up.  us per step of the TMEM kernel against fixed 32 planes: FP32-shift 64^3
// 13.4 / 68.8, 96^3 42 / 80, 128^3 84 / 87, 160^3 168 / 183, 192^3 268 / 272, 256^3 621 / 627;
// FP16 96^3 29 / 68, 128^3 61 / 67, 160^3 121 / 139, 256^3 442 / 450.
// keep: a depth that stays unless another ends 5 % earlier (0: none).
inline int segment_planes(long long columns, int nz, int slots, int keep = 0)
{
    auto schedule_end = [&](int seg) {  // in half planes
        const long long nseg = (nz + seg - 1) / seg, len = 2 * seg + 5, last = 2 * (nz - (nseg - 1) * seg) + 5;
        // the full segments launch first, then one last segment per column
        const long long full = (nseg - 1) * columns, rem = full % slots, t0 = (full / slots) * len;
        long long end = t0 + std::max(rem ? len : 0, (columns + slots - 1) / slots * last);
        while ((slots - rem) * ((end - t0) / last) + rem * (end - t0 >= len ? (end - t0 - len) / last : 0) < columns)
            ++end;
        return end;
    };
    int best = 1;
    long long best_end = -1;
    for (int seg = nz < 64 ? nz : 64; seg >= 1; --seg) {
        const long long end = schedule_end(seg);
        if (best_end < 0 || end < best_end) {
            best = seg;
            best_end = end;
        }
    }
    return keep > 0 && keep <= nz && schedule_end(keep) * 95 <= best_end * 100 ? keep : best;
}

// ... of a launch over solver s in tiles of tile_x x tile_y columns, per_sm blocks
// resident on an SM (kept in the solver: the grid and its tiles do not change).  Two
// blocks share an SM's memory traffic, which the schedule does not see: 192 x 200 x 192
// FP32-shift in 32 x 8 tiles takes 457 us with its 48 planes, 427 with 32 (2 % apart in
// the schedule), while 160 x 168 x 160 gains 3 % (schedule 7 %) and 96 x 104 x 96 16 %
// (55 %), so there 32 planes stay unless the schedule ends 5 % earlier.
inline int solver_segment_planes(const Solver& s, int tile_x, int tile_y, int per_sm)
{
    int& seg = s.seg_planes[per_sm == 1 ? 0 : 1];
    if (seg == 0)
        seg = segment_planes((long long)((s.nx + tile_x - 1) / tile_x) * ((s.ny + tile_y - 1) / tile_y), s.nz,
                             per_sm * (s.num_sms > 0 ? s.num_sms : 152), per_sm == 1 ? 0 : 32);
    return seg;
}

// Programmatic dependent launch.  A kernel launched after this one with the
// programmatic-serialization attribute may be scheduled once every block of
// this one has signalled (pdl_release, at the top of the kernel); its blocks
// run their prologue and then stop in pdl_wait until this kernel has finished
// and its memory operations are visible.  Without the attribute pdl_wait
// returns at once.
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch `kernel` with the programmatic-serialization attribute (outside a
// stream capture; inside one, as an ordinary launch).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                       Args&&... args)
{
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(st, &cap);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cap == cudaStreamCaptureStatusNone ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// Raise kernel K's dynamic shared-memory limit to `bytes`, once per device
// and process.
template <auto K>
cudaError_t set_smem_limit_once(int bytes)
{
    static std::atomic<unsigned long long> done{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_acq_rel);
    return e;
}

__device__ __forceinline__ int wrapi(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }
__device__ __forceinline__ int modi(int v, int n) { return ((v % n) + n) % n; }

template <int ST>
__device__ __forceinline__ float raw_value(const StepParams& p, typename Storage<ST>::T v, int i)
{
    using S = Storage<ST>;
    const float f = S::load(&v);
    return S::shifted ? f : f - p.bw[i] * p.rho_ref;
}

// Whole 32 x 8 tiles with 16-byte aligned rows.
template <int ST>
bool single_fast_ok(const Solver& s)
{
    using T = typename Storage<ST>::T;
    return s.nx % kTileX == 0 && s.ny % kTileY == 0 && (s.nx * (int)sizeof(T)) % 16 == 0;
}

}  // namespace elbm
