"""GPU: the 128-key attention kernel with its first copies in front (two row tiles and chunks of up to 22 blocks of the table's width,
or a single row tile; test_chunk_plan_rounds.py has which plans take which order) and behind the bounds check and zeros: both sides of the line against the fp64 checker, and the same bits."""
import numpy as np
import pytest

import oracle
from gpu_util import check_attention, gpu_attention
from test_gpu_attention_tiles import in_table_of, problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,Hq,Hkv", [(19, 14, 2), (9, 14, 2)])
@pytest.mark.parametrize("chunks", [1, 2, 5])
@pytest.mark.parametrize("lens", [(0, 1, 64), (63, 65, 400), (129, 1344, 700)])
def test_both_sides_of_the_line(monkeypatch, lens, chunks, T, Hq, Hkv):
    monkeypatch.setenv("SDV_TEST_CHUNKS", str(chunks))
    p = problem(sum(lens) + T, lens, T=T, Hq=Hq, Hkv=Hkv)
    p.n_nodes = np.array([T, max(1, T - 1), 2], dtype=np.int32)
    ref, rlse = oracle.attention(oracle.Geometry.of(p), p.k_cache, p.v_cache, p.q, p.k_tree, p.v_tree, p.scale)
    ok = np.isfinite(rlse)
    first = None
    for width in (22 * chunks, 22 * chunks + 1):              # two row tiles: in front, behind; one: in front both times
        out, lse, status = gpu_attention(in_table_of(p, width))
        assert status == 0
        check_attention(out[ok], ref[ok], f"lens={lens} chunks={chunks} width={width}")
        np.testing.assert_allclose(lse[ok], rlse[ok], rtol=2e-3, atol=2e-3)
        for b in range(3):
            assert (out[b, p.n_nodes[b]:] == 0).all() and (lse[b, p.n_nodes[b]:] == 0).all()
        if first is None:
            first = out, lse
    np.testing.assert_array_equal(first[0], out)
    np.testing.assert_array_equal(first[1], lse)
