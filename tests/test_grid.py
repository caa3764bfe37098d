"""Grids of the fused launches (csrc/dilbm_grid.h, host arithmetic).

A small program is compiled with the header and prints the grids of a range of
lattices; the rules are checked here by their statement."""
import os
import subprocess

import pytest

from paper_2106_08950_gb300 import build as B

SRC = r"""
#include <cstdio>
#include "dilbm_grid.h"
using namespace dilbm;
int main() {
    const long long items[] = {1, 3, 8, 100, 400, 1517, 1518, 1519, 1822, 2048, 4096, 8192, 32768, 65536, 131072, 131073};
    const long long parts[] = {0, 1, 7, 32, 33, 64, 256, 512, 1056, 2048, 84000};
    const int fits[][2] = {{2, 10}, {4, 5}, {8, 2}, {2, 12}, {4, 6}, {8, 3}, {4, 1}};
    for (long long i : items)
        for (long long p : parts)
            for (auto &f : fits)
                for (int bps : {0, 1, 3})
                    for (int sms : {1, 152}) {
                        const SweepShape sh{f[0], bps};
                        const FusedGrid g = fused_grid(i, p, f[0], f[1], sms, sh);
                        std::printf("%lld %lld %d %d %d %d %lld %d %d\n", i, p, f[0], f[1], bps, sms, g.blocks, g.pblocks,
                                    (int)one_item_per_warp(i, p, f[0], f[1], sms, sh));
                    }
}
"""


@pytest.fixture(scope="module")
def grids(tmp_path_factory):
    d = tmp_path_factory.mktemp("grid")
    (d / "grid.cpp").write_text(SRC)
    exe = str(d / "grid")
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-Werror", "-I", B.CSRC, str(d / "grid.cpp"), "-o", exe])
    return [tuple(map(int, ln.split())) for ln in subprocess.check_output([exe]).decode().splitlines()]


def test_one_grid_holds_its_own_particle_blocks(grids):
    """All blocks fit the device, some sweep, and the particle blocks are the
    rule's for the segments and the occupancy that this grid was made for."""
    assert len(grids) == 16 * 11 * 7 * 3 * 2
    for items, parts, w, per_sm, bps, sms, blocks, pblocks, _ in grids:
        most = sms * (min(bps, per_sm) if bps else per_sm)
        each = min(max(items // (4 * most * w), 1), 8)              # particles of a warp
        share = most * 2 * parts // (2 * parts + items)             # a particle's update as two segments
        want = min(-(-parts // (w * each)), max(most // 10, share, 1))
        assert pblocks == want
        assert blocks - pblocks >= 1
        assert blocks <= max(most, 2)                               # (one of each kind at least)
        assert blocks - pblocks <= -(-items // w)


def test_one_item_per_warp_counts_the_same_grids_sweeping_blocks(grids):
    for items, parts, w, per_sm, bps, sms, blocks, pblocks, one in grids:
        assert bool(one) == (items <= (blocks - pblocks) * w)


def test_a_launch_takes_both_counts_from_one_grid():
    """The launchers set the particle blocks from the grid that they launch,
    after any trial of another one."""
    src = open(os.path.join(B.CSRC, "dilbm_launch.cuh")).read()
    assert src.count("const FusedGrid g = fused_grid(") == src.count("p, &run, g, ") == 2
    assert src.count("run->pblocks = g.pblocks;") == 1 and src.count("dim3 blocks((unsigned)g.blocks)") == 1
    assert "run.pblocks" not in src
