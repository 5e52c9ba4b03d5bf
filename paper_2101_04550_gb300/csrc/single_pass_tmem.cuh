// Single-pass step with two population arrays: TMA-fed, warp-specialised, with
// the populations parked in tensor memory (TMEM) between their two uses.
//
// The per-node arithmetic is that of single_pass.cuh (bit-identical results).
// A block of five warpgroups owns a tile of 64 x 8 or 32 x 16 columns and marches
// through a segment of z planes (segment_planes()):
//   * the first warp of warpgroup 4 loads plane k of the tile with one 4-D
//     TMA box (x, y, z 1, population 27) into a ring of one or two tile buffers in
//     shared memory, and the ring of nodes around the tile -- two TMA row
//     boxes and the two columns by cp.async -- into a ring of two
//     buffers; one mbarrier per buffer ("full") tracks both kinds of copy.
//     Its other three warps compute the anomaly of the ring: the row below, the
//     row above, the two columns (TMEM lane quarters follow a warp's rank within its
//     warpgroup, so the consumers must make whole warpgroups);
//   * the 16 warps of warpgroups 0..3 own 32 nodes of the tile each.  For plane k a
//     thread reads its node's 27 populations from shared memory once, hands
//     the buffer back ("empty" mbarrier), parks the values in its TMEM lane,
//     computes the anomaly Q~ of its node, publishes it ("qready")
//     and relaxes plane k-1 -- with the values parked one plane earlier --
//     once every warp has published the anomaly of plane k-1 (the central
//     difference of Eq. Paastar1 needs the face neighbours), pushing the 27
//     results with coalesced stores.
// A tile buffer comes back as soon as it has been read, and the relaxation of the
// previous plane covers the next load.  There is no block-wide barrier in the loop.
//
// What bounds it: FP32 storage the memory system, with pushes that straddle tile
// edges (see launch_single_tmem()); 16-bit storage instruction issue, 736
// instructions a node (824 before the relaxation took the populations in pairs and
// the pushes one pointer per c_x; FP32 663, before 763), issued on 72 % of the cycles.
// Every wait is bounded (2 s, or as soon as another thread of the block gave
// up); a wait that gives up sets ELBM_ERR_TIMEOUT in the status word, and the
// block winds down: the loader waits, again bounded, for the copies in flight,
// and the TMEM is freed by the warp that allocated it.
#pragma once
#include "relax_pairs.cuh"
#include "single_pass_tma.cuh"

namespace elbm {

constexpr int kTmTileY = 16;                      // rows of the 32-wide tile (one consumer warp each)
constexpr int kTmConsumers = kTileX * kTmTileY;   // 512 threads, a node of the tile each
constexpr int kTmWarps = kTmConsumers / 32;
constexpr int kTmThreads = kTmConsumers + 128;    // + the loading warpgroup
// Registers per thread of the walls-and-force kernel: the block is launched with
// kTmLaunchRegs for everyone (what its size leaves of the SM's), and the loading
// warpgroup gives up what the consumers take, never more than that (channel 512 x 128 x
// 256 FP32: 728 us per step without, 663 with; the periodic kernel needs no more
// than 96 and FP16 runs 1.6 % slower with the split).
constexpr int kTmLaunchRegs = 96, kTmLoaderRegs = 64, kTmConsumerRegs = 104;
static_assert(kTmConsumers * kTmConsumerRegs + 128 * kTmLoaderRegs <= kTmThreads * kTmLaunchRegs,
              "the consumers must not wait for registers that the block does not own");
template <int N>
__device__ __forceinline__ void setmaxnreg_dec()
{
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void setmaxnreg_inc()
{
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}
constexpr uint32_t kTmTmemCols = 256;             // 2 plane slots x 4 warps per lane quarter x 32

// TX: tile width, 32 (x 16 rows) or 64 (x 8 rows); NT: tile buffers; PB: how a tile
// is loaded -- 0 by TMA (whole tiles), else by cp.async in pieces of 16 or 4 bytes
// (any grid).
template <int ST, int TX, int NT, int PB = 0>
struct TmemLayout {
    using T = typename Storage<ST>::T;
    static constexpr int es = (int)sizeof(T);
    static constexpr int TY = kTmConsumers / TX;
    static constexpr int ntile = NT;
    static constexpr int ring_warps = 3;  // spare warps of the loading warpgroup, for the ring's anomaly
    // elements a row takes; 16-bit rows in 4-byte words start in either half of one
    static constexpr bool words = PB == 4 && es == 2;
    static constexpr int RS = words ? TX + 2 : TX;
    static constexpr int tile_bytes = (27 * TY * RS * es + 127) / 128 * 128;  // one plane of the tile
    static constexpr int row_box_bytes = 27 * RS * es;               // one ring row, all populations
    static constexpr int row_stride = (row_box_bytes + 127) / 128 * 128;
    static constexpr int ncol = 2 * TY;                        // ring column nodes
    static constexpr int cols_bytes = 27 * ncol * 4;                 // as 4-byte words
    static constexpr int qx_bytes = TY * (TX + 2) * 4;
    static constexpr int qy_bytes = (TY + 2) * TX * 4;
    // the ring's anomaly in units of one warp: TX / 32 for the row below, as many
    // for the row above, one for the two columns
    static constexpr int row_units = TX / 32, ring_units = 2 * row_units + 1;
    static constexpr int off_tile = 0;                               // [ntile] planes
    static constexpr int off_rows = off_tile + ntile * tile_bytes;   // [2 slots][2 sides]
    static constexpr int off_cols = off_rows + 4 * row_stride;       // [2 slots]
    static constexpr int off_qx = off_cols + 2 * cols_bytes;         // [kTmaQSlots]
    static constexpr int off_qy = off_qx + kTmaQSlots * qx_bytes;
    static constexpr int off_bar = (off_qy + kTmaQSlots * qy_bytes + 7) / 8 * 8;
    // mbarriers, in this order: full and empty per tile buffer, full and empty
    // per ring buffer, one per anomaly slot
    static constexpr int bar_full_t = 0, bar_empty_t = ntile, bar_full_r = 2 * ntile, bar_empty_r = 2 * ntile + 2;
    static constexpr int bar_qready = 2 * ntile + 4;
    static constexpr int nbar = bar_qready + kTmaQSlots;
    static constexpr int off_abort = off_bar + 8 * nbar;
    static constexpr int off_tmem = off_abort + 4;
    static constexpr int bytes = off_abort + 16 + 128;               // + slack for aligning the base
    static_assert(PB != 0 || tile_bytes == 27 * kTmConsumers * es, "tile boxes must keep 128-byte alignment");
};

// One tile column of a single-pass step: the TX x 512/TX columns at (x0, y0),
// planes z0 .. z1-1, from p.f into dst; every thread of the block takes part.
// tm_tile / tm_row are the tensor maps of p.f (kernel parameters, or device
// memory made visible to the tensor-map proxy).  smem_raw is the block's
// dynamic shared memory (TmemLayout<ST, TX, NT>::bytes).
// BC: walls (half-way bounce-back below y = 0 and above y = ny-1, with the
// anomaly's negated ghost value in the central difference) and the body force,
// read from the parameter block as in the two-pass kernels; with neither set
// in p it computes the same bits as BC = false.
// PB != 0: the grid may be any; the tile's last columns and rows beyond it are
// idle, the ring closes around the ones it has, and the four warps of the loading
// warpgroup copy the tile and its ring with cp.async, a quarter of the populations
// each (no tensor maps: rows need not start on 16 bytes).
template <int ST, int TX, int NT, bool BC, bool FX = false, int PB = 0>
__device__ __forceinline__ void tmem_tile_step(const CUtensorMap* tm_tile, const CUtensorMap* tm_row,
                                               const StepParams& p, void* dst, int x0, int y0, int z0, int z1,
                                               unsigned char* smem_raw)
{
    using S = Storage<ST>;
    using T = typename S::T;
    using L = TmemLayout<ST, TX, NT, PB>;
    constexpr int TY = L::TY, RS = L::RS;
    // columns and rows of the tile that the grid has
    const int w = PB == 0 ? TX : min(TX, p.nx - x0), h = PB == 0 ? TY : min(TY, p.ny - y0);
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t sbase = (raw_addr + 127u) & ~127u;
    unsigned char* base = smem_raw + (sbase - raw_addr);
    const uint32_t bar0 = sbase + L::off_bar;
    auto full_t = [&](int b) { return bar0 + 8u * (L::bar_full_t + b); };
    auto empty_t = [&](int b) { return bar0 + 8u * (L::bar_empty_t + b); };
    auto full_r = [&](int r) { return bar0 + 8u * (L::bar_full_r + r); };
    auto empty_r = [&](int r) { return bar0 + 8u * (L::bar_empty_r + r); };
    auto qready = [&](int s) { return bar0 + 8u * (L::bar_qready + s); };
    volatile int* abort_flag = reinterpret_cast<volatile int*>(base + L::off_abort);

    const int K = (z1 - z0) + 2;  // planes z0-1 .. z1
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int kLoader = kTmConsumers / 32;  // first warp of the loading warpgroup
    pdl_release();

    // Every thread arrives for itself (one arrival per warp behind __syncwarp() was
    // no faster in FP32 and 2.8 % slower in FP16, 256^3)
    if (threadIdx.x == 0) {
        for (int b = 0; b < L::ntile; ++b) {
            mbar_init(full_t(b), PB == 0 ? 1 : 128);  // expect_tx, or the loaders' cp.async arrivals
            mbar_init(empty_t(b), kTmConsumers);
        }
        for (int r = 0; r < 2; ++r) {
            // lane 0's expect_tx and the cp.async arrivals of the loading warp, or of the four
            mbar_init(full_r(r), PB == 0 ? 1 + 32 : 128);
            mbar_init(empty_r(r), 32 * L::ring_warps);
        }
        for (int s = 0; s < kTmaQSlots; ++s) mbar_init(qready(s), kTmConsumers + 32 * L::ring_warps);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kLoader) {
        tmem_alloc(sbase + L::off_tmem, kTmTmemCols);
        tmem_relinquish();
    }
    tmem_fence_before_sync();
    __syncthreads();
    tmem_fence_after_sync();
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(base + L::off_tmem);
    pdl_wait();  // the previous step has written the source array

    // bounded in time (kTmaWaitNs), or as soon as another thread of the block gave up
    auto wait = [&](uint32_t bar, unsigned parity) { return bounded_wait(bar, parity, abort_flag, p.status, kTmaWaitNs); };
    auto drain = [&](uint32_t bar, unsigned parity) { bounded_drain(bar, parity, kTmaWaitNs); };
    auto plane_of = [&](int k) { return wrapi(z0 - 1 + k, p.nz); };
    float* qxs = reinterpret_cast<float*>(base + L::off_qx);
    float* qys = reinterpret_cast<float*>(base + L::off_qy);
    auto QX = [&](int s, int y, int x) -> float& { return qxs[(s * TY + y) * (TX + 2) + x]; };
    auto QY = [&](int s, int y, int x) -> float& { return qys[(s * (TY + 2) + y) * TX + x]; };
    // 16-bit rows copied as 4-byte words: element index of the row's first node (all
    // populations alike up to i N), and the half word population i starts in
    auto row_start = [&](int k, int y) { return plane_of(k) * p.plane + y * p.nx + x0; };
    auto half_of = [&](int i, int start) { return L::words ? (start + (i & 1) * p.N) & 1 : 0; };
    // unit u of the ring's anomaly of plane k (one warp)
    auto ring_unit = [&](int u, int k) {
        const int r = k & 1, s = k % kTmaQSlots;
        auto anomaly_of = [&](auto&& gval, float* q) {
            float drho, j[3];
            moments_of<3>(p, gval, drho, j);
            const float inv_rho = 1.0f / (p.rho_ref + drho);
#pragma unroll
            for (int a = 0; a < 3; ++a) q[a] = anomaly(p, a, j[a], j[a] * inv_rho);
        };
        float qh[3];
        if (u < 2 * L::row_units) {
            const int side = u / L::row_units, x = (u % L::row_units) * 32 + lane;
            const T* row = reinterpret_cast<const T*>(base + L::off_rows + (2 * r + side) * L::row_stride) + x;
            const int start = L::words ? row_start(k, side ? wrapi(y0 + h, p.ny) : wrapi(y0 - 1, p.ny)) : 0;
            anomaly_of([&](int i) { return raw_value<ST>(p, row[i * RS + half_of(i, start)], i); }, qh);
            if (PB == 0 || x < w) QY(s, side ? h + 1 : 0, x) = qh[1];
        } else if (lane < L::ncol && (PB == 0 || (lane & (TY - 1)) < h)) {
            const unsigned* cols = reinterpret_cast<const unsigned*>(base + L::off_cols + r * L::cols_bytes) + lane;
            const int y = lane & (TY - 1), cx = lane < TY ? wrapi(x0 - 1, p.nx) : wrapi(x0 + w, p.nx);
            const int idx0 = plane_of(k) * p.plane + (y0 + y) * p.nx + cx;
            anomaly_of([&](int i) { return stage_value<ST>(p, cols[i * L::ncol], (i * p.N + idx0) & 1, i); }, qh);
            QX(s, y, lane < TY ? 0 : w + 1) = qh[0];
        }
    };

    if (warp >= kLoader) {
        if (BC) setmaxnreg_dec<kTmLoaderRegs>();
        const int duty = warp - kLoader - 1;  // ring anomaly: 0 the row below the tile, 1 the row above, 2 the two columns
        auto ring_plane = [&](int k) {
            if (k > 0 && k < K - 1) {
                if (duty == 2) {
                    ring_unit(L::ring_units - 1, k);
                } else {
                    for (int u = 0; u < L::row_units; ++u) ring_unit(duty * L::row_units + u, k);
                }
            }
            __syncwarp();
            mbar_arrive(empty_r(k & 1));
            mbar_arrive(qready(k % kTmaQSlots));
        };
        // ring column node kk: x0-1 for kk < TY, x0+w for kk >= TY, row y0 + kk % TY
        const int ylo = wrapi(y0 - 1, p.ny), yhi = wrapi(y0 + h, p.ny);
        const int cxl = wrapi(x0 - 1, p.nx), cxr = wrapi(x0 + w, p.nx);
        auto load_columns = [&](int zk, int r) {
            unsigned* cols = reinterpret_cast<unsigned*>(base + L::off_cols + r * L::cols_bytes);
            for (int c = PB == 0 ? lane : (int)threadIdx.x - kTmConsumers; c < 27 * L::ncol; c += PB == 0 ? 32 : 128) {
                const int i = c / L::ncol, kk = c % L::ncol, y = PB == 0 ? kk & (TY - 1) : min(kk & (TY - 1), h - 1);
                const int idx = i * p.N + zk * p.plane + (y0 + y) * p.nx + (kk < TY ? cxl : cxr);
                cp_async4(cols + c, stage_src<ST>(p, idx));
            }
            cp_async_mbar_arrive(full_r(r));
        };
        int issued = 0;
        if constexpr (PB != 0) {
            // A row goes over in pieces of PB bytes, 16-bit rows on 4-byte pieces in the words
            // that hold them: lane l takes pieces l, l + 32, ... of the tile's rows of a
            // population and of its two ring rows, warp q populations q, q + 4, ...  Where a
            // piece lies is the same in every plane and population, so it is worked out once,
            // and the copies of a population are independent instructions.
            constexpr int NPR = PB == 16 ? TX * L::es / 16 : L::es == 4 ? TX : TX / 2 + 1;  // pieces of a row
            constexpr int EP = PB == 16 ? 16 / L::es : 1;                                   // elements of a piece
            constexpr int NT_TILE = (TY * NPR + 31) / 32, NT_RING = (2 * NPR + 31) / 32;
            // first element of the piece (words: of its row) in a plane, or -1 where the
            // grid has none; its byte among the population's rows in the buffer
            struct Piece {
                int from, to;
            };
            auto piece = [&](int c, int row, bool any, int stride) {
                const int x = c % NPR * EP;
                return Piece{any && (L::words || x < w) ? row * p.nx + x0 + (L::words ? 0 : x) : -1,
                             c / NPR * stride + c % NPR * PB};
            };
            Piece tile_piece[NT_TILE], ring_piece[NT_RING];
#pragma unroll
            for (int q = 0; q < NT_TILE; ++q) {
                const int c = lane + 32 * q;
                tile_piece[q] = piece(c, y0 + c / NPR, c / NPR < h, RS * L::es);
            }
#pragma unroll
            for (int q = 0; q < NT_RING; ++q) {
                const int c = lane + 32 * q;
                ring_piece[q] = piece(c, c / NPR ? yhi : ylo, c / NPR < 2, L::row_stride);
            }
            // piece c of a row of the population that starts at element i N + plane
            auto copy = [&](unsigned char* to, const Piece& q, int c, int start) {
                if constexpr (PB == 16) {
                    if (q.from >= 0) cp_async16(to + q.to, static_cast<const T*>(p.f) + start + q.from);
                } else if constexpr (L::es == 4) {
                    if (q.from >= 0)
                        cp_async4(reinterpret_cast<unsigned*>(to + q.to), static_cast<const T*>(p.f) + start + q.from);
                } else {
                    const int at = start + q.from, j = c % NPR;
                    if (q.from >= 0 && j < ((at & 1) + w + 1) >> 1)
                        cp_async4(reinterpret_cast<unsigned*>(to + q.to), static_cast<const unsigned*>(p.f) + (at >> 1) + j);
                }
            };
            for (int k = 0; k < K; ++k) {
                const int b = k % L::ntile, r = k & 1, zk = plane_of(k);
                bool ok = true;
                if (k >= L::ntile) ok = wait(empty_t(b), ((k / L::ntile) - 1) & 1);
                if (ok && k >= 2) ok = wait(empty_r(r), ((k / 2) - 1) & 1);
                if (!__all_sync(0xffffffffu, ok)) break;
                for (int i = warp - kLoader; i < 27; i += 4) {
                    unsigned char* to = base + L::off_tile + b * L::tile_bytes + i * TY * RS * L::es;
#pragma unroll
                    for (int q = 0; q < NT_TILE; ++q) copy(to, tile_piece[q], lane + 32 * q, i * p.N + zk * p.plane);
                }
                cp_async_mbar_arrive(full_t(b));
                issued = k + 1;
                for (int i = warp - kLoader; i < 27; i += 4) {
                    unsigned char* to = base + L::off_rows + 2 * r * L::row_stride + i * RS * L::es;
#pragma unroll
                    for (int q = 0; q < NT_RING; ++q) copy(to, ring_piece[q], lane + 32 * q, i * p.N + zk * p.plane);
                }
                load_columns(zk, r);
                if (warp != kLoader && k > 0) {  // the ring of the plane before, while this one is on its way
                    if (!__all_sync(0xffffffffu, wait(full_r(r ^ 1), ((k - 1) / 2) & 1))) break;
                    ring_plane(k - 1);
                }
            }
            if (warp != kLoader && issued == K && __all_sync(0xffffffffu, wait(full_r((K - 1) & 1), ((K - 1) / 2) & 1)))
                ring_plane(K - 1);
            cp_async_wait_all();
            __syncwarp();
        } else if (warp == kLoader) {
            // ---------------------------------------------------- loader
            for (int k = 0; k < K; ++k) {
                const int b = k % L::ntile, r = k & 1;
                bool ok = true;
                if (k >= L::ntile) ok = wait(empty_t(b), ((k / L::ntile) - 1) & 1);
                if (ok && k >= 2) ok = wait(empty_r(r), ((k / 2) - 1) & 1);
                if (!__all_sync(0xffffffffu, ok)) break;
                const int zk = plane_of(k);
                if (lane == 0) {
                    mbar_arrive_expect_tx(full_t(b), L::tile_bytes);
                    tma_load_4d(sbase + L::off_tile + b * L::tile_bytes, tm_tile, x0, y0, zk, 0, full_t(b));
                    mbar_arrive_expect_tx(full_r(r), 2 * L::row_box_bytes);
                    tma_load_4d(sbase + L::off_rows + (2 * r) * L::row_stride, tm_row, x0, ylo, zk, 0, full_r(r));
                    tma_load_4d(sbase + L::off_rows + (2 * r + 1) * L::row_stride, tm_row, x0, yhi, zk, 0,
                                full_r(r));
                }
                load_columns(zk, r);
                issued = k + 1;
            }
            cp_async_wait_all();
            // no copy may still be in flight when the block retires
            if (lane == 0) {
                for (int k = max(0, issued - L::ntile); k < issued; ++k) drain(full_t(k % L::ntile), (k / L::ntile) & 1);
                for (int k = max(0, issued - 2); k < issued; ++k) drain(full_r(k & 1), (k / 2) & 1);
            }
            __syncwarp();
        } else {
            // ------------------------------------------------ ring anomaly
            for (int k = 0; k < K; ++k) {
                if (!__all_sync(0xffffffffu, wait(full_r(k & 1), (k / 2) & 1))) break;
                ring_plane(k);
            }
        }
    } else {
        // ------------------------------------------------------ consumers
        if (BC) setmaxnreg_inc<kTmConsumerRegs>();
        const int tx = threadIdx.x & (TX - 1), ty = threadIdx.x / TX;
        const int gx = x0 + tx, gy = y0 + ty;
        const T* tile = reinterpret_cast<const T*>(base + L::off_tile);
        auto anomaly_m = [&](auto&& gval, float* q, float& drho, float* j, float& inv_rho) {
            moments_of<3>(p, gval, drho, j);
            inv_rho = 1.0f / (p.rho_ref + drho);
#pragma unroll
            for (int a = 0; a < 3; ++a) q[a] = anomaly(p, a, j[a], j[a] * inv_rho);
        };
        // TMEM columns of this thread: its warp's lane quarter; 32 columns per
        // warp of the quarter (warps w, w+4, w+8, w+12 share a quarter); 128 per plane slot
        const uint32_t t_own = tmem_base + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((warp >> 2) * 32);
        T* out = static_cast<T*>(dst);
        // push target of population i = (cx, cy, cz): one pointer per cx, which stays
        // over the march, and one 32-bit element offset per (cy, cz)
        T* const xp[3] = {out + (gx == 0 ? p.nx - 1 : gx - 1), out + p.N + gx,
                          out + 2 * p.N + (gx == p.nx - 1 ? 0 : gx + 1)};
        const int yo[3] = {(gy == 0 ? p.ny - 1 : gy - 1) * p.nx, 3 * p.N + gy * p.nx,
                           6 * p.N + (gy == p.ny - 1 ? 0 : gy + 1) * p.nx};
        constexpr int kPlaneElems = TY * RS;  // stride between populations in a tile buffer
        const bool active = PB == 0 || (tx < w && ty < h);

        float qz_prev = 0.f, qz_cur = 0.f;
        // moments of the own node of the plane relaxed next (computed with its anomaly)
        float m_drho = 0.f, m_j[3] = {0.f, 0.f, 0.f}, m_inv_rho = 1.f;
        for (int k = 0; k < K; ++k) {
            const int b = k % L::ntile, s = k % kTmaQSlots;
            if (!__all_sync(0xffffffffu, wait(full_t(b), (k / L::ntile) & 1))) break;
            float q[3], k_drho, k_j[3], k_inv_rho;
            {
                const T* own = tile + b * (L::tile_bytes / L::es) + ty * RS + tx;
                const int start = L::words ? row_start(k, gy) : 0;
                float g[27];  // in pair order
#pragma unroll
                for (int i = 0; i < 27; ++i) g[pair_slot(i)] = raw_value<ST>(p, own[i * kPlaneElems + half_of(i, start)], i);
                // the parking store (unused for the outer two planes) takes every value, so
                // the reads are complete when the buffer goes back; an arrival right behind
                // the loads can overtake them where they queue behind the loader's copies,
                // and the refill then lands under them
                tmem_store27(t_own + (uint32_t)((k & 1) * 128), g);
                mbar_arrive(empty_t(b));
                anomaly_m([&](int i) { return g[pair_slot(i)]; }, q, k_drho, k_j, k_inv_rho);
            }
            if (active) {
                QX(s, ty, tx + 1) = q[0];
                QY(s, ty + 1, tx) = q[1];
            }
            __syncwarp();
            mbar_arrive(qready(s));
            if (k == 0) {
                qz_prev = q[2];
                continue;
            }
            if (k == 1) {
                qz_cur = q[2];
                m_drho = k_drho;
                m_inv_rho = k_inv_rho;
#pragma unroll
                for (int a = 0; a < 3; ++a) m_j[a] = k_j[a];
                continue;
            }
            // relax plane k-1 (z = z0 + k - 2) once every warp has published its anomaly
            const float qz_next = q[2];
            const int kc = k - 1, sc = kc % kTmaQSlots;
            if (!__all_sync(0xffffffffu, wait(qready(sc), (kc / kTmaQSlots) & 1))) break;
            float g[27];
            tmem_wait_st();
            tmem_load27(t_own + (uint32_t)((kc & 1) * 128), g);
            const float drho = m_drho, j[3] = {m_j[0], m_j[1], m_j[2]};  // moments_of of the same values
            float d[3] = {0.f, 0.f, 0.f};
            if (p.eq_mode == 0) {
                d[0] = (QX(sc, ty, tx + 2) - QX(sc, ty, tx)) * p.inv_2lam[0];
                float qyp = QY(sc, ty + 2, tx), qym = QY(sc, ty, tx);
                if (BC && p.walls_y && gy == p.ny - 1) qyp = -QY(sc, ty + 1, tx);  // ghost beyond the wall
                if (BC && p.walls_y && gy == 0) qym = -QY(sc, ty + 1, tx);
                d[1] = (qyp - qym) * p.inv_2lam[1];
                d[2] = (qz_next - qz_prev) * p.inv_2lam[2];
            }
            const int z = z0 + k - 2;
            const int zo[3] = {wrapi(z - 1, p.nz) * p.plane, 9 * p.N + z * p.plane,
                               18 * p.N + wrapi(z + 1, p.nz) * p.plane};
            int yz[9];  // push target: element offset of the row (y + cy, z + cz) of population (-1, cy, cz)
#pragma unroll
            for (int c = 0; c < 9; ++c) yz[c] = yo[c % 3] + zo[c / 3];
            auto put = [&](int i, float gn) {
                const float v = S::shifted ? gn : fmaf(p.bw[i], p.rho_ref, gn);
                if (BC && p.walls_y && ((cy_of(i) == 1 && gy == p.ny - 1) || (cy_of(i) == -1 && gy == 0))) {
                    // half-way bounce-back: f'_i returns reversed to its own node, as
                    // population opp(i), stored against opp(i)'s baseline
                    const float vb = S::shifted ? v + bounce_rebase<3>(p, 26 - i) : v;
                    S::store(out + opaque((26 - i) * p.N) + gx + gy * p.nx + z * p.plane, vb);
                } else {
                    S::store(xp[cx_of(i) + 1] + yz[i / 3], v);
                }
            };
            // (the walls-and-force kernel recomputes 1/rho: one register fewer across the loop)
            if (active) relax_pairs<BC, FX>(p, g, put, drho, j, d, BC ? 1.0f / (p.rho_ref + drho) : m_inv_rho);
            qz_prev = qz_cur;
            qz_cur = qz_next;
            m_drho = k_drho;
            m_inv_rho = k_inv_rho;
#pragma unroll
            for (int a = 0; a < 3; ++a) m_j[a] = k_j[a];
        }
        tmem_wait_st();
    }
    // every TMEM access of the block is complete before the loader frees it
    tmem_fence_before_sync();
    __syncthreads();
    if (warp == kLoader) {
        tmem_fence_after_sync();
        tmem_dealloc(tmem_base, kTmTmemCols);
    }
}

// The single-pass step of one grid: block (bx, by, bz) takes the tile column
// at (TX bx, 512/TX by), planes seg bz onwards.  FX (with BC): the body
// force acts along x alone.
template <int ST, int TX, int NT, bool BC = false, bool FX = false>
__global__ void __launch_bounds__(kTmThreads, 1)
    k_single_pass_tmem(const __grid_constant__ CUtensorMap tm_tile, const __grid_constant__ CUtensorMap tm_row,
                       const __grid_constant__ StepParams p, void* dst, int seg)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int z0 = blockIdx.z * seg;
    tmem_tile_step<ST, TX, NT, BC, FX>(&tm_tile, &tm_row, p, dst, blockIdx.x * TX, blockIdx.y * (kTmConsumers / TX), z0,
                                   min(p.nz, z0 + seg), smem_raw);
}

template <int ST>
bool single_tmem_ok(const Solver& s, const void* src, const void* dst)
{
    using T = typename Storage<ST>::T;
    return s.nx % kTileX == 0 && s.ny % kTmTileY == 0 && (s.nx * (int)sizeof(T)) % 16 == 0 &&
           ((uintptr_t)src % 16 == 0) && ((uintptr_t)dst % 16 == 0);
}

// A kernel that moves registers between its warpgroups must be launched with
// kTmLaunchRegs a thread, or its consumers would wait for registers the block does
// not own: checked once per kernel and device.
template <auto K>
cudaError_t check_launch_registers()
{
    static std::atomic<unsigned long long> done{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
    cudaFuncAttributes a;
    e = cudaFuncGetAttributes(&a, K);
    if (e == cudaSuccess && (a.numRegs + 7) / 8 * 8 < kTmLaunchRegs) e = cudaErrorInvalidConfiguration;
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_acq_rel);
    return e;
}

template <int ST, int TX, int NT, bool BC, bool FX>
cudaError_t launch_single_tmem_tile(const Solver& s, const StepParams& p, void* dst, bool* launched)
{
    *launched = false;
    if (!single_tmem_ok<ST>(s, p.f, dst)) return cudaSuccess;
    CUtensorMap tm_tile, tm_row;
    constexpr int TY = kTmConsumers / TX;
    if (encode_population_maps(s, p.f, TX, TY, &tm_tile, &tm_row) != cudaSuccess) return cudaSuccess;
    const int smem = TmemLayout<ST, TX, NT>::bytes;
    cudaError_t e = set_smem_limit_once<k_single_pass_tmem<ST, TX, NT, BC, FX>>(smem);
    if (e == cudaSuccess && BC) e = check_launch_registers<k_single_pass_tmem<ST, TX, NT, BC, FX>>();
    if (e != cudaSuccess) return e;
    const int seg = solver_segment_planes(s, TX, TY, 1);
    const dim3 grid((unsigned)(s.nx / TX), (unsigned)(s.ny / TY), (unsigned)((s.nz + seg - 1) / seg));
    // programmatic dependent launch helps the 16-bit form at every size (256^3
    // +0.5 %) and the FP32 form on short steps (32^3 10.3 -> 7.3 us, 128^3 94.4 ->
    // 92.9, 160^3 187.0 -> 186.4); from 192^3 on it costs that form 0.2-0.7 %
    if (sizeof(typename Storage<ST>::T) == 2 || s.N <= 4ll << 20) {
        e = launch_pdl(k_single_pass_tmem<ST, TX, NT, BC, FX>, grid, dim3(kTmThreads), smem, s.stream, tm_tile, tm_row, p,
                       dst, seg);
    } else {
        k_single_pass_tmem<ST, TX, NT, BC, FX><<<grid, kTmThreads, smem, s.stream>>>(tm_tile, tm_row, p, dst, seg);
        e = cudaGetLastError();
    }
    *launched = e == cudaSuccess;
    return e;
}

// Tile shape and buffers.  64-wide tiles wherever nx allows: a push along x leaves
// 32-byte sectors at the tile's edges half written by one SM and half by another,
// half as many of them on 64-wide tiles (a plain copy of 27 shifted populations at
// 256^3 runs at 5.4 TB/s in 32-wide tiles, 6.1 in 64-wide ones, 6.7 unshifted).
// A second tile buffer keeps a load in flight while the first one is read; in FP32
// its 55 KB come out of the L1 cache, which merges the pushes of a row's two warps,
// so only the 64-wide periodic form gains at every size, the others on grids that a
// few planes per block cover.  us per step, one against two buffers: 256^3 FP32
// 64-wide 643 / 617, 32-wide 679 / 734; channel 512 x 128 x 256 FP32 672 / 712;
// 64^3 14.6 / 12.9, 32^3 7.1 / 6.5.  (Before: 32-wide tiles, one buffer, the ring's
// anomaly on the consumers: 682; FP16 32-wide 485, now 440.)
template <int ST, bool BC = false, bool FX = false>
cudaError_t launch_single_tmem(const Solver& s, const StepParams& p, void* dst, bool* launched)
{
    constexpr bool wide_storage = sizeof(typename Storage<ST>::T) == 4;
    if (s.nx % 64 == 0) return launch_single_tmem_tile<ST, 64, wide_storage && BC ? 1 : 2, BC, FX>(s, p, dst, launched);
    if (wide_storage && s.N > 1 << 18) return launch_single_tmem_tile<ST, 32, 1, BC, FX>(s, p, dst, launched);
    return launch_single_tmem_tile<ST, 32, 2, BC, FX>(s, p, dst, launched);
}

// One single-pass step from s.f into dst (D3Q27 only; the caller swaps the arrays):
// the TMA-fed kernels where the geometry allows (whole tiles with TMEM, else 32 x 8
// tiles), else the cp.async-fed TMEM one (single_pass_ragged.cu).
template <int D>
cudaError_t step_single_impl(const Solver& s, void* dst, long long* launches)
{
    if constexpr (D != 3) {
        (void)s;
        (void)dst;
        (void)launches;
        return cudaErrorNotSupported;
    } else {
        StepParams p;
        fill_params(s, p);
        p.parity = 0;
        cudaError_t e = cudaSuccess;
        ELBM_DISPATCH_STORAGE(s.storage, {
            bool done = false;
            if (p.walls_y || p.forced) {
                // walls and body force: the TMEM form only (the caller checks its geometry);
                // a force along x alone (or none) takes the lighter force increment
                const bool fx = p.g[1] == 0.f && p.g[2] == 0.f;
                e = fx ? launch_single_tmem<ST, true, true>(s, p, dst, &done)
                       : launch_single_tmem<ST, true, false>(s, p, dst, &done);
                if (e == cudaSuccess && !done) e = cudaErrorNotSupported;
                if (e == cudaSuccess) ++*launches;
                return e;
            }
            e = launch_single_tmem<ST>(s, p, dst, &done);
            if (e == cudaSuccess && !done) e = launch_single_tma<ST>(s, p, dst, &done);
            if (e == cudaSuccess && !done) e = launch_single_ragged(s, p, dst);
        });
        if (e != cudaSuccess) return e;
        ++*launches;
        return cudaSuccess;
    }
}

}  // namespace elbm
