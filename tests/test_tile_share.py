"""The split of a call's tiles over the CTAs of a persistent kernel (TilePlan, TileShare), run on the host: the shares that are launched hold
every tile once, in order, none is empty, none is more than two tiles longer than an even split's, and none holds tiles of two lambda
rows where the rows can have shares of their own within that length; shares beyond those launched would hold nothing."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_05699_b200", "csrc")
SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "kvq_device.cuh"
int main()
{
    srand(1);
    for (long it = 0; it < 200000; ++it) {
        const long n_seg = 1 + rand() % (it % 3 ? 12 : 400), rpl = 1 + rand() % (it % 2 ? 400 : 9000), segs = 1 + rand() % (it % 5 ? 1 : 20);
        const unsigned parts = 1 + rand() % 150;
        const int rows = it % 7 ? 128 : 256;
        const long tps = (rpl + rows - 1) / rows, tiles = n_seg * tps, even = (tiles + parts - 1) / parts;
        const long row_tiles = (segs < n_seg ? segs : n_seg) * tps, n_rows = (tiles + row_tiles - 1) / row_tiles;
        const bool apart = n_rows <= (long)parts && (n_rows == 1 || (row_tiles + (long)parts / n_rows - 1) / ((long)parts / n_rows) <= even + 2);
        const kvq::TilePlan plan(n_seg, rpl, parts, rows, segs);
        long at = 0;
        for (unsigned p = 0; p < parts || p < plan.shares; ++p) {
            const kvq::TileShare s(plan, p);
            if ((s.n > 0) != (p < plan.shares) || plan.shares > parts) {
                printf("n_seg %ld rpl %ld segs %ld parts %u: %u shares, share %u has %d tiles\n", n_seg, rpl, segs, parts, plan.shares, p, s.n);
                return 1;
            }
            if (s.n == 0) continue;
            if (s.tps != tps || s.seg != (unsigned)(at / tps) || s.tin != (unsigned)(at % tps) || s.begin != at || s.n < 0 || s.n > even + 2) {
                printf("n_seg %ld rpl %ld segs %ld parts %u: share %u begins at %ld (%ld), %d tiles of %ld\n", n_seg, rpl, segs, parts, p,
                       (long)s.begin, at, s.n, even);
                return 1;
            }
            if (apart && s.begin / row_tiles != (s.begin + s.n - 1) / row_tiles) {
                printf("n_seg %ld rpl %ld segs %ld parts %u: share %u (%d tiles from %ld) crosses a lambda row of %ld tiles\n", n_seg, rpl, segs,
                       parts, p, s.n, (long)s.begin, row_tiles);
                return 1;
            }
            at += s.n;
        }
        if (at != tiles) {
            printf("n_seg %ld rpl %ld segs %ld parts %u: %ld of %ld tiles\n", n_seg, rpl, segs, parts, at, tiles);
            return 1;
        }
    }
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="no nvcc")
def test_every_tile_belongs_to_one_share(tmp_path):
    src, exe = tmp_path / "share.cu", tmp_path / "share"
    src.write_text(SOURCE)
    subprocess.run(["nvcc", "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_100a,code=sm_100a", "-I", CSRC, "-o", str(exe), str(src)],
                   check=True, capture_output=True, text=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout
