"""How an LM-head call is dealt out (csrc/lmhead_plan.cuh), compiled for the host: tiles cut into pieces are covered once, and W
is brought to L2 ahead where that was measured to be faster and not where it was slower."""
import os
import subprocess

import pytest

from paper_2509_18824_b200 import build

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "lmhead_plan.cuh"
using namespace sdv;
static int cover() {                                       // every (tile, chunk) once, and columns that the kernel takes
    long checks = 0;
    for (int rows = 1; rows <= 512; ++rows) {
        const LmColumns c = lm_columns(rows);
        if (c.part_n % 16 || c.part_n > 256 || c.padded() < rows || c.padded() > 512 || (c.n_parts == 2) != (rows > 256)) { printf("rows %d\n", rows); return 1; }
    }
    for (int n_pad = 288; n_pad <= 512; n_pad += 32)
        for (int pairs : {1, 2, 35, 37, 71, 74})
            for (int tiles = 1; tiles <= 700; ++tiles, ++checks) {
                const LmSlices s = plan_slices(tiles, pairs, n_pad);
                const int n_chunks = (n_pad + 31) / 32;
                const bool cut = s.slices > 0;
                if (s.rounds != tiles / pairs) { printf("rounds %d %d %d\n", n_pad, pairs, tiles); return 1; }
                if (cut && (s.slices * s.slice_chunks < n_chunks || (s.slices - 1) * s.slice_chunks >= n_chunks || s.slice_chunks > 8)) { printf("pieces %d %d %d\n", n_pad, pairs, tiles); return 1; }
                if (cut == (tiles % pairs == 0) && cut) { printf("nothing left %d %d %d\n", n_pad, pairs, tiles); return 1; }
            }
    printf("%ld\n", checks);
    return 0;
}
int main(int argc, char** argv) {
    if (argc == 1) return cover();
    printf("%d\n", (int)brings_ahead(atoi(argv[1]), (atoi(argv[2]) + 255) / 256, 74));
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    nvcc = build._nvcc()
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("lmhead_plan")
    (d / "plan.cu").write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_100a,code=sm_100a", "-I", build.INCLUDE, "-I", build.CSRC,
                    str(d / "plan.cu"), "-o", str(d / "plan")], check=True)
    return lambda *a: subprocess.run([str(d / "plan"), *map(str, a)], capture_output=True, text=True, check=True).stdout.strip()


def test_pieces_cover_the_tiles(plan):
    assert int(plan()) == 8 * 6 * 700


@pytest.mark.parametrize("Hd,V,ahead", [(4096, 32000, 1), (2048, 50257, 1), (768, 32000, 1), (3584, 152064, 1), (1024, 1025, 1), (128, 6000, 1),
                                        (512, 6000, 0), (512, 4099, 0), (384, 6000, 0), (256, 6000, 0)])
def test_k_steps_brought_to_l2(plan, Hd, V, ahead):
    assert int(plan(Hd, V)) == ahead
