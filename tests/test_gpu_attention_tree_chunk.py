"""GPU: sequences whose last key chunk holds the tree's keys alone (36 cache blocks in seven chunks, 41, 42, 48 and 56 in eight), and
ones with a few blocks beside the tree or split evenly, against the fp64 checker."""
import numpy as np
import pytest

import oracle
from gpu_util import check_attention, gpu_attention
from test_gpu_attention_tiles import problem

pytestmark = pytest.mark.gpu


def blocks_of_last_chunk(blocks, chunks, tree=3, start=5):
    """Cache blocks beside the tree in the last chunk, as csrc/attention_shared.cuh cuts a sequence."""
    even = -(-blocks // chunks)
    counted = blocks + (tree if even > start and (blocks - 1) % even + 1 >= start else 0)
    per = -(-counted // chunks)
    used = max(2, -(-counted // per))
    return max(0, blocks - (used - 1) * per), used


@pytest.mark.parametrize("T,Hq,Hkv", [(19, 14, 2), (2, 8, 1), (64, 4, 2)])
@pytest.mark.parametrize("blocks,chunks,beside", [(22, 4, 4), (28, 5, 4), (36, 7, 0), (37, 7, 1), (41, 8, 0), (42, 8, 0), (48, 8, 0), (56, 8, 0)])
def test_last_chunk_of_the_tree_alone(monkeypatch, blocks, chunks, beside, T, Hq, Hkv):
    assert blocks_of_last_chunk(blocks, chunks) == (beside, chunks)
    monkeypatch.setenv("SDV_TEST_CHUNKS", str(chunks))
    lens = (64 * blocks, 64 * blocks - 63, 64 * blocks - 1)
    p = problem(blocks + T, lens, T=T, Hq=Hq, Hkv=Hkv)
    p.n_nodes = np.array([T, max(1, T - 1), 1], dtype=np.int32)
    out, lse, status = gpu_attention(p)
    assert status == 0
    ref, rlse = oracle.attention(oracle.Geometry.of(p), p.k_cache, p.v_cache, p.q, p.k_tree, p.v_tree, p.scale)
    ok = np.isfinite(rlse)
    check_attention(out[ok], ref[ok], f"blocks={blocks} chunks={chunks}")
    np.testing.assert_allclose(lse[ok], rlse[ok], rtol=2e-3, atol=2e-3)
    for b in range(3):
        assert (out[b, p.n_nodes[b]:] == 0).all() and (lse[b, p.n_nodes[b]:] == 0).all()
