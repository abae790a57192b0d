"""The split of a sequence into key chunks where the tree's keys, in the last chunk, count for several cache blocks
(csrc/attention_shared.cuh), compiled for the host: the chunks cover the sequence once, the last is shorter by what the
tree counts for, and sequences whose chunks hold at most kStartBlocks, or whose last one is shorter than that anyway, are
cut as without a tree."""
import os
import subprocess

import pytest

from paper_2509_18824_b200 import build

SOURCE = r"""
#include <cstdio>
#include "attention_shared.cuh"
using namespace sdv;
int main() {
    const int wholes[] = {-1, 0, 5, 10};
    long checks = 0;
    for (int n = 1; n <= kMaxChunks; ++n)
        for (int whole : wholes)
            for (int blocks = 0; blocks <= 3000; ++blocks, ++checks) {
                AttnPlan plain, p;
                plain.set_chunks(n, whole);
                p.set_chunks(n, whole);
                p.tree_blocks = kTreeBlocks;
                const int len = blocks * kBlock;
                const ChunkRange first = chunk_range(p, len, 4000, 0), was = chunk_range(plain, len, 4000, 0);
                const int even = (blocks + n - 1) / n;
                int left = blocks;                                     // of the last chunk that an even split uses
                while (left > even) left -= even;
                const bool counts = n > 1 && blocks > whole && blocks > n * kStartBlocks && left >= kStartBlocks;
                bool ok = first.tiles_total == blocks && first.n_chunks >= 1 && first.n_chunks <= n;
                if (!counts) ok = ok && first.tpc == was.tpc && first.n_chunks == was.n_chunks;
                else ok = ok && first.tpc == (blocks + kTreeBlocks + n - 1) / n && first.n_chunks * first.tpc >= blocks + kTreeBlocks;
                int at = 0;
                for (int k = 0; k < n; ++k) {
                    const ChunkRange r = chunk_range(p, len, 4000, k);
                    ok = ok && r.n_chunks == first.n_chunks && r.tpc == first.tpc && r.t0 == at && r.t1 >= r.t0 && r.t1 - r.t0 <= r.tpc;
                    if (counts && k == first.n_chunks - 1) ok = ok && r.t1 - r.t0 <= r.tpc - kTreeBlocks;
                    at = r.t1;
                    if (k == first.n_chunks - 1) ok = ok && at == blocks;
                }
                if (!ok) { printf("n %d whole %d blocks %d\n", n, whole, blocks); return 1; }
            }
    printf("%ld\n", checks);
}
"""


def test_last_chunk_is_shorter_by_the_tree(tmp_path):
    src, exe = tmp_path / "chunks.cu", tmp_path / "chunks"
    src.write_text(SOURCE)
    nvcc = build._nvcc()
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_100a,code=sm_100a", "-I", build.INCLUDE, "-I", build.CSRC,
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 90000
