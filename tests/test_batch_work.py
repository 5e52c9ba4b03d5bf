"""The work list of the flattened single-pass batch covers every plane of every
tile column once, also on grids with more than 2^15 and 2^16 planes."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2101_04550_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "batch_work.h"
int main(int argc, char** argv)  // tile_y seg interleaved [nx ny nz]...
{
    std::vector<elbm::WorkGrid> grids;
    for (int k = 4; k + 2 < argc; k += 3) grids.push_back({atoi(argv[k]), atoi(argv[k + 1]), atoi(argv[k + 2])});
    for (const auto& w : elbm::work_list(grids, 32, atoi(argv[1]), atoi(argv[2]), atoi(argv[3]) != 0))
        std::printf("%d %d %d %d %d\n", w.member, w.x0, w.y0, w.z0, w.z0 + w.planes);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("work")
    src, exe = str(d / "w.cpp"), str(d / "w")
    with open(src, "w") as fh:
        fh.write(PROGRAM)
    subprocess.check_call([cxx, "-std=c++17", "-O1", "-I", build.CSRC, src, "-o", exe])
    assert os.path.exists(exe)
    return exe


@pytest.mark.parametrize("tile_y,seg", [(16, 32), (16, 16), (8, 8)])
@pytest.mark.parametrize("interleaved", [0, 1])
def test_every_plane_once(program, tile_y, seg, interleaved):
    grids = [(64, 32, 33), (32, 16, 32767), (32, 16, 32768), (32, 16, 65537), (32, 16, 150000), (96, 48, 3)]
    args = [str(v) for v in (tile_y, seg, interleaved)] + [str(v) for g in grids for v in g]
    out = subprocess.check_output([program] + args, text=True)
    items = np.array(out.split(), dtype=np.int64).reshape(-1, 5)
    for m, (nx, ny, nz) in enumerate(grids):
        mine = items[items[:, 0] == m]
        count = np.zeros((ny // tile_y, nx // 32, nz + 1), dtype=np.int64)
        for _, x0, y0, z0, z1 in mine:
            assert x0 % 32 == 0 and y0 % tile_y == 0 and 0 <= z0 < z1 <= nz and z1 - z0 <= seg
            count[y0 // tile_y, x0 // 32, z0] += 1
            count[y0 // tile_y, x0 // 32, z1] -= 1
        assert (np.cumsum(count, axis=2)[:, :, :nz] == 1).all()
    assert ((0 <= items[:, 0]) & (items[:, 0] < len(grids))).all()
    if interleaved:  # one item of each grid first
        assert items[:len(grids), 0].tolist() == list(range(len(grids)))
    else:
        assert (np.diff(items[:, 0]) >= 0).all()
