"""The split of a sequence into key chunks (csrc/attention_shared.cuh), compiled for the host: for every number of cache
blocks, every cluster size and every way of planning, the chunks cover the sequence once and are as few and as short
as stated."""
import os
import subprocess

import pytest

from paper_2509_18824_b200 import build

SOURCE = r"""
#include <cstdio>
#include "attention_shared.cuh"
using namespace sdv;
static int fail(const char* what, int n, int whole, int blocks) { printf("%s: n %d whole %d blocks %d\n", what, n, whole, blocks); return 1; }
static int check(int n, int whole, int blocks, int table) {
    AttnPlan p;
    p.set_chunks(n, whole);
    const int len = blocks == 0 ? 0 : (blocks - 1) * kBlock + 1 + blocks % kBlock;
    const int there = blocks < table ? blocks : table;                 // (a length beyond the table is cut off there)
    const ChunkRange first = chunk_range(p, len, table, 0);
    const int c = first.n_chunks, per = (there + n - 1) / n;
    if (first.tiles_total != there || c < 1 || c > n) return fail("count", n, whole, blocks);
    int at = 0;
    for (int k = 0; k < n; ++k) {                                      // CTAs behind the last chunk have nothing
        const ChunkRange r = chunk_range(p, len, table, k);
        if (r.n_chunks != c || r.tpc != first.tpc || r.t0 != at || r.t1 < r.t0 || r.t1 - r.t0 > r.tpc) return fail("cover", n, whole, blocks);
        at = r.t1;
        if (k == c - 1 && at != there) return fail("end", n, whole, blocks);
    }
    if (there == 0 || n == 1 || there <= whole) return c == 1 && first.tpc == there ? 0 : fail("whole", n, whole, blocks);
    if (first.tpc != per) return fail("longest", n, whole, blocks);
    if (whole < 0) return c == n ? 0 : fail("all", n, whole, blocks);
    return (c == 2 || (c - 1) * per < there) && c * per >= there ? 0 : fail("fewest", n, whole, blocks);
}
int main() {
    const int wholes[] = {-1, 0, 5, 10}, far[] = {1 << 20, (1 << 25) - 9, (1 << 25) - 2};
    long checks = 0;
    for (int n = 1; n <= kMaxChunks; ++n)
        for (int whole : wholes) {
            for (int blocks = 0; blocks <= 20000; ++blocks, ++checks)
                if (check(n, whole, blocks, 1 << 25) || check(n, whole, blocks, blocks < 1 ? 1 : blocks) || check(n, whole, blocks, 37)) return 1;
            for (int b0 : far)
                for (int blocks = b0; blocks < b0 + 2; ++blocks, ++checks)
                    if (check(n, whole, blocks, 1 << 25)) return 1;
        }
    printf("%ld\n", checks);
}
"""


def test_chunks_cover_a_sequence_once(tmp_path):
    src, exe = tmp_path / "chunks.cu", tmp_path / "chunks"
    src.write_text(SOURCE)
    nvcc = build._nvcc()
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_100a,code=sm_100a", "-I", build.INCLUDE, "-I", build.CSRC,
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 600000
