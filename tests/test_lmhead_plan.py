"""How an LM-head call is dealt out (csrc/lmhead_plan.cuh), compiled for the host: tiles cut into pieces are covered once, and two
row blocks share a launch where that was measured to be faster and not where it was slower."""
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
                if (s.rounds != tiles / pairs || s.cost < s.rounds || s.cost > s.rounds + 1.0) { printf("cost %d %d %d\n", n_pad, pairs, tiles); return 1; }
                if (cut && (s.slices * s.slice_chunks < n_chunks || (s.slices - 1) * s.slice_chunks >= n_chunks || s.slice_chunks > 8)) { printf("pieces %d %d %d\n", n_pad, pairs, tiles); return 1; }
                if (cut == (tiles % pairs == 0) && cut) { printf("nothing left %d %d %d\n", n_pad, pairs, tiles); return 1; }
            }
    printf("%ld\n", checks);
    return 0;
}
int main(int argc, char** argv) {
    if (argc == 1) return cover();
    if (argc == 3) { printf("%d\n", (int)brings_ahead(atoi(argv[1]), (atoi(argv[2]) + 255) / 256, 74)); return 0; }
    const int M = atoi(argv[1]), V = atoi(argv[2]), Hd = atoi(argv[3]);       // how the row blocks of a call share launches, 74 pairs
    const int n = (M + 511) / 512, rows = ((M + n - 1) / n + 15) / 16 * 16;
    for (int rb = 0; rb < n;) {
        const bool two = rb + 1 < n && side_by_side(rows, M - (rb + 1) * rows < rows ? M - (rb + 1) * rows : rows, Hd, (V + 255) / 256, 74);
        printf("%d", two ? 2 : 1);
        rb += two ? 2 : 1;
    }
    printf("\n");
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


# "2": side by side, "11": one behind the other.  Measured where the comment at side_by_side says so.
@pytest.mark.parametrize("M,V,Hd,launches", [
    (544, 152064, 3584, "2"), (600, 152064, 3584, "2"), (960, 152064, 3584, "2"), (1025, 152064, 3584, "21"),
    (600, 128256, 4096, "2"), (960, 128256, 4096, "2"), (513, 50257, 2048, "2"), (960, 50257, 2048, "2"), (2048, 32000, 4096, "22"),
    (513, 4099, 1024, "2"), (600, 200, 1024, "2"), (1537, 4099, 3584, "22"),
    # a second block whose own columns are fewer, where W's tiles take many rounds
    (513, 152064, 3584, "11"), (513, 152064, 1024, "11"), (520, 128256, 4096, "11"), (528, 94000, 3584, "11"), (513, 110000, 3584, "11"),
    (577, 128256, 4096, "11"), (769, 128256, 4096, "11"), (961, 128256, 4096, "11"), (1537, 128256, 4096, "211")])
def test_row_blocks_share_a_launch_where_it_is_faster(plan, M, V, Hd, launches):
    assert plan(M, V, Hd) == launches


@pytest.mark.parametrize("Hd,V,ahead", [(4096, 32000, 1), (2048, 50257, 1), (768, 32000, 1), (3584, 152064, 1), (1024, 1025, 1), (128, 6000, 1),
                                        (512, 6000, 0), (512, 4099, 0), (384, 6000, 0), (256, 6000, 0)])
def test_k_steps_brought_to_l2(plan, Hd, V, ahead):
    assert int(plan(Hd, V)) == ahead
