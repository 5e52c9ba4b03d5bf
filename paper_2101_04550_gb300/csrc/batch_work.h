// Work list of the flattened single-pass batch (batch_single.cuh): which block takes
// which planes of which tile column of which member.  Plain C++, host and device.
#pragma once
#include <algorithm>
#include <cstddef>
#include <vector>

namespace elbm {

// Planes z0 .. z0 + planes - 1 of the tile column at (x0, y0) of a member.  The
// member's index and the planes of a segment are small (a batch holds at most 40
// members); coordinates take whole words, since a grid may have more than 2^15 planes.
struct alignas(16) WorkItem {
    short member, planes;
    int x0, y0, z0;
};
static_assert(sizeof(WorkItem) == 16, "one 16-byte load per block");

struct WorkGrid {
    int nx, ny, nz;
};

// Items of every grid in columns of tile_x x tile_y and segments of at most seg planes:
// grid after grid, or (interleaved) one item of each grid in turn.
inline std::vector<WorkItem> work_list(const std::vector<WorkGrid>& grids, int tile_x, int tile_y, int seg,
                                       bool interleaved)
{
    std::vector<std::vector<WorkItem>> per(grids.size());
    std::size_t longest = 0;
    for (std::size_t m = 0; m < grids.size(); ++m) {
        const WorkGrid& g = grids[m];
        for (int z0 = 0; z0 < g.nz; z0 += seg)
            for (int y0 = 0; y0 < g.ny; y0 += tile_y)
                for (int x0 = 0; x0 < g.nx; x0 += tile_x)
                    per[m].push_back({(short)m, (short)std::min(g.nz - z0, seg), x0, y0, z0});
        longest = std::max(longest, per[m].size());
    }
    std::vector<WorkItem> work;
    if (!interleaved) {
        for (const auto& v : per) work.insert(work.end(), v.begin(), v.end());
    } else {
        for (std::size_t k = 0; k < longest; ++k)
            for (const auto& v : per)
                if (k < v.size()) work.push_back(v[k]);
    }
    return work;
}

}  // namespace elbm
