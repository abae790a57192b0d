"""The number of key chunks of an attention launch (csrc/attention_plan.cuh), compiled for the host: a launch whose row tiles
fit one round goes in several only where an SM then works through a fifth fewer blocks, however wide the block table is."""
import os
import subprocess

import pytest

from paper_2509_18824_b200 import build

SOURCE = r"""
#include <cstdio>
#include "attention_plan.cuh"
using namespace sdv;
int main() {
    const int sms = 148, lost[] = {0, 1, 3};                           // clusters that do not find their SMs side by side
    const int widths[] = {1, 2, 6, 17, 33, 65, 129, 257, 433, 434, 512, 831, 832, 1024, 2048, 4096, 16384, 1 << 20, 1 << 25};
    long checks = 0;
    for (int less : lost)
        for (int base = 1; base <= sms; ++base) {
            auto resident = [&](int c) { return c == 1 ? sms : sms / c - (c > 2 ? less : 0); };
            auto rounds = [&](int c) { return (base + resident(c) - 1) / resident(c); };
            int most = 0;
            for (int c = 1; c <= kMaxChunks; ++c) if (rounds(c) == 1) most = c;
            for (int blocks : widths) {
                AttnPlan p;
                if (!choose_wide(&p, base, blocks, sms, 0, resident)) { printf("base %d blocks %d: 64-key kernel\n", base, blocks); return 1; }
                const int n = p.n_chunks, r = rounds(n);
                if (r > 1 && 5 * r * most > 4 * n) { printf("base %d blocks %d: %d chunks in %d rounds, %d fit one\n", base, blocks, n, r, most); return 1; }
                if ((p.whole_blocks < 0) != (r > 1)) { printf("base %d blocks %d: whole %d\n", base, blocks, p.whole_blocks); return 1; }
                ++checks;
            }
            for (int c = 1; c <= kMaxChunks; ++c) {                    // the test hook asks for any number
                AttnPlan p;
                if (choose_wide(&p, base, 512, sms, c, resident) && p.n_chunks != c) { printf("base %d: forced %d\n", base, c); return 1; }
            }
        }
    AttnPlan p;                                                        // 128 row tiles: whole, in every table
    for (int blocks = 1; blocks <= 5000; ++blocks, ++checks)
        if (!choose_wide(&p, 128, blocks, sms, 0, [](int c) { return 148 / c; }) || p.n_chunks != 1) { printf("128: %d\n", blocks); return 1; }
    printf("%ld\n", checks);
}
"""


def test_a_wider_table_does_not_bring_several_rounds(tmp_path):
    src, exe = tmp_path / "rounds.cu", tmp_path / "rounds"
    src.write_text(SOURCE)
    nvcc = build._nvcc()
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_100a,code=sm_100a", "-I", build.INCLUDE, "-I", build.CSRC,
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 13000


FIRST_COPIES = r"""
#include <cstdio>
#include <cstdlib>
#include "attention_plan.cuh"
using namespace sdv;
int main(int argc, char** argv) {                          // B, KV heads, row tiles, width of the table
    const int B = atoi(argv[1]), Hkv = atoi(argv[2]), blocks = atoi(argv[4]), sms = 148;
    AttnPlan p;
    p.row_tiles = atoi(argv[3]);
    const int base = B * Hkv * p.row_tiles;
    if (!choose_wide(&p, base, blocks, sms, 0, [&](int c) { return c <= 2 ? sms / c : c < 7 ? sms / c - 1 : 15; })) { printf("64\n"); return 0; }
    p.ranked = B > 1 && B <= 64 && base * p.n_chunks > sms;
    printf("%d %d\n", p.n_chunks, (int)copies_first(p, blocks));
}
"""


@pytest.fixture(scope="module")
def first_copies(tmp_path_factory):
    nvcc = build._nvcc()
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("first_copies")
    (d / "first.cu").write_text(FIRST_COPIES)
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_100a,code=sm_100a", "-I", build.INCLUDE, "-I", build.CSRC,
                    str(d / "first.cu"), "-o", str(d / "first")], check=True)
    return lambda *a: subprocess.run([str(d / "first"), *map(str, a)], capture_output=True, text=True, check=True).stdout.split()


# (chunks, whether the first copies go first), as measured where the comment at copies_first says so
@pytest.mark.parametrize("B,Hkv,row_tiles,blocks,plan", [
    (1, 4, 4, 2, (1, 1)), (1, 4, 4, 33, (4, 1)), (1, 4, 4, 129, (6, 1)), (1, 4, 4, 251, (6, 0)),
    (8, 4, 4, 22, (1, 1)), (8, 4, 4, 23, (1, 0)), (8, 4, 4, 65, (1, 0)), (4, 4, 4, 34, (2, 1)), (4, 4, 4, 36, (2, 0)), (4, 4, 4, 43, (2, 0)),
    (3, 4, 4, 41, (3, 0)), (2, 4, 4, 17, (3, 1)), (2, 4, 4, 87, (4, 1)), (8, 4, 2, 43, (2, 1)), (16, 4, 2, 25, (1, 0)),
    (8, 4, 1, 65, (4, 1)), (8, 4, 1, 200, (4, 1)), (37, 4, 1, 16, (1, 1)),
    # several rounds, of one and of more row tiles, more sequences than are ranked by length, and one sequence
    (72, 4, 1, 65, (1, 0)), (100, 4, 1, 32, (1, 0)), (1, 64, 4, 64, (1, 0)), (16, 4, 4, 257, (1, 0))])
def test_first_copies_go_first(first_copies, B, Hkv, row_tiles, blocks, plan):
    assert tuple(int(x) for x in first_copies(B, Hkv, row_tiles, blocks)) == plan
