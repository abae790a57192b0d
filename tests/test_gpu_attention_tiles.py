"""GPU: attention at the edges of the 128-key tiles and key chunks (odd and even block counts, half tiles,
sequences of one batch cut into different numbers of chunks), and scores that rise so far above the first
tile's that the rows' reference has to be raised, through both kernels."""
import copy

import numpy as np
import pytest
import torch

import oracle
from paper_2509_18824_b200 import binding as sd
from paper_2509_18824_b200 import workloads as wl
from paper_2509_18824_b200.step import to_device
from helpers import Tiny
from gpu_util import gpu_attention, check_attention

pytestmark = pytest.mark.gpu


def problem(seed, lens, T=19, Hq=14, Hkv=2, gain=3.0):
    g = np.random.default_rng(seed)
    B = len(lens)
    par = np.stack([np.array([-1] + [int(g.integers(0, i)) for i in range(1, T)]) for _ in range(B)])
    return Tiny(seed, B=B, T=T, Hq=Hq, Hkv=Hkv, D=128, lens=lens, parents=par, gain=gain)


@pytest.mark.parametrize("chunks", [0, 1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("lens", [(0, 64, 129), (128, 127, 385), (640, 511, 1), (1023, 257, 130), (1409, 1024, 66)])
def test_tile_and_chunk_edges(monkeypatch, lens, chunks):
    """19 nodes x 7 heads = a row tile of 126 rows and one of 7."""
    monkeypatch.setenv("SDV_TEST_CHUNKS", str(chunks))
    p = problem(sum(lens), lens)
    p.n_nodes = np.array([19, 18, 5], dtype=np.int32)
    out, lse, status = gpu_attention(p)
    assert status == 0
    ref, rlse = oracle.attention(oracle.Geometry.of(p), p.k_cache, p.v_cache, p.q, p.k_tree, p.v_tree, p.scale)
    ok = np.isfinite(rlse)
    check_attention(out[ok], ref[ok], f"lens={lens} chunks={chunks}")
    np.testing.assert_allclose(lse[ok], rlse[ok], rtol=2e-3, atol=2e-3)
    for b in range(3):
        assert (out[b, p.n_nodes[b]:] == 0).all() and (lse[b, p.n_nodes[b]:] == 0).all()


def rising(seed):
    """Keys that grow from block to block: the scores of later tiles lie hundreds of powers of two above the
    first tile's."""
    p = problem(seed, (900, 333, 1000), T=12, Hq=8, Hkv=2, gain=1.0)
    for b in range(p.B):
        for j in range(int(p.len[b]) // 64 + 1):
            blk = p.block_table[b, j]
            x = wl.bf16_bits_to_f32(p.k_cache[blk]) * np.float32(1.0 + 60.0 * ((j * 5) % 8))
            p.k_cache[blk] = wl.f32_to_bf16_bits(x)
    return p


@pytest.mark.parametrize("layers", [1, 40])
def test_reference_is_raised(layers):
    """One layer runs the 128-key kernel, forty layers of this size the 64-key kernel."""
    p = rising(77)
    ref, rlse = oracle.attention(oracle.Geometry.of(p), p.k_cache, p.v_cache, p.q, p.k_tree, p.v_tree, p.scale)
    if layers == 1:
        out, lse, status = gpu_attention(p)
        outs, lses = [out], [lse]
    else:
        bt, st = sd.Batch.of(p), sd.new_status()
        sd.sd_tree_prepare(bt, st)
        kc, vc, q, kt, vt = (to_device(x) for x in (p.k_cache, p.v_cache, p.q, p.k_tree, p.v_tree))
        o = [torch.full((p.B, p.T_max, p.Hq, p.D), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(layers)]
        ls = [torch.zeros((p.B, p.T_max, p.Hq), dtype=torch.float32, device="cuda") for _ in range(layers)]
        ws = torch.empty(sd.sd_workspace_bytes(bt), dtype=torch.uint8, device="cuda")
        sd.sd_verify_attention_layers(bt, sd.AttentionLayerSet([kc] * layers, [vc] * layers, [q] * layers, [kt] * layers,
                                                               [vt] * layers, o, ls), float(p.scale), ws, st)
        torch.cuda.synchronize()
        status = int(st.item())
        outs, lses = [x.float().cpu().numpy() for x in (o[0], o[-1])], [x.cpu().numpy() for x in (ls[0], ls[-1])]
    assert status == 0
    for out, lse in zip(outs, lses):
        rel = np.linalg.norm(out - ref) / np.linalg.norm(ref)
        assert rel <= 2e-2, rel
        np.testing.assert_allclose(lse, rlse, rtol=2e-3, atol=2e-3)


@pytest.mark.parametrize("stale", [0, -7, 333, 5000, 2**31 - 1])
def test_lengths_written_by_the_kernel_ahead(stale):
    """An attention call may begin while the kernel ahead still runs, and looks at the lengths then: whatever
    stands there must not matter once that kernel (here acceptance, which writes them) has finished."""
    p = problem(5, (900, 333, 1000))
    ref, ref_lse, status = gpu_attention(p)
    assert status == 0
    bt, src = sd.Batch.of(p), sd.Batch.of(p)
    src.len -= 1                                          # one node accepted: the length of p
    st = sd.new_status()
    sd.sd_tree_prepare(bt, st)
    i32 = lambda *shape: torch.zeros(shape, dtype=torch.int32, device="cuda")
    draft, argmax, n_acc, path, tok = i32(p.B, p.T_max) + 1, i32(p.B * p.T_max), i32(p.B), i32(p.B, p.T_max), i32(p.B, p.T_max)
    cache = sd.kv_layer(to_device(p.k_cache), to_device(p.v_cache))
    q, kt, vt = to_device(p.q), to_device(p.k_tree), to_device(p.v_tree)
    ws = torch.empty(sd.sd_workspace_bytes(bt), dtype=torch.uint8, device="cuda")
    for _ in range(8):
        out = torch.full((p.B, p.T_max, p.Hq, p.D), 7.0, dtype=torch.bfloat16, device="cuda")
        lse = torch.zeros((p.B, p.T_max, p.Hq), dtype=torch.float32, device="cuda")
        bt.len.fill_(stale)
        sd.sd_accept_tree(src, draft, argmax, n_acc, path, tok, bt.len, st)
        sd.sd_verify_attention(bt, cache, q, kt, vt, float(p.scale), out, lse, ws, st)
        torch.cuda.synchronize()
        assert int(st.item()) == 0 and (n_acc == 1).all()
        np.testing.assert_array_equal(out.float().cpu().numpy(), ref)
        np.testing.assert_array_equal(lse.cpu().numpy(), ref_lse)


def in_table_of(p, width):
    """The same problem in a block table of that width (as a server keeps it); nothing may look behind the sequences."""
    q = copy.copy(p)
    q.block_table = np.full((p.B, width), 1 << 20, dtype=np.int32)
    q.block_table[:, :p.block_table.shape[1]] = p.block_table
    q.max_blocks = width
    return q


@pytest.mark.parametrize("lens", [(2048,), (700, 2300), (4000, 130, 1000)])
def test_split_follows_the_length_and_not_the_table(monkeypatch, lens):
    p = problem(sum(lens), lens)
    cut = {}
    for chunks in range(1, 9):
        monkeypatch.setenv("SDV_TEST_CHUNKS", str(chunks))
        out, lse, status = gpu_attention(p)
        assert status == 0
        for width in (200, 512):                          # the same bits whatever the width
            wide, wide_lse, status = gpu_attention(in_table_of(p, width))
            assert status == 0
            np.testing.assert_array_equal(wide, out)
            np.testing.assert_array_equal(wide_lse, lse)
        cut[chunks] = out
    monkeypatch.delenv("SDV_TEST_CHUNKS")
    out, _, status = gpu_attention(in_table_of(p, 512))
    assert status == 0
    b = int(np.argmax(lens))                              # unforced: the long sequence is cut into as many chunks as pay
    same = [c for c in cut if np.array_equal(out[b], cut[c][b])]
    assert same and max(same) >= 4, same


@pytest.mark.parametrize("blocks", [0, 1, 5, 6, 10, 11, 12])
@pytest.mark.parametrize("B", [1, 8, 37])
def test_short_sequences_in_a_wide_table(blocks, B):
    """Around the lengths from which a sequence is cut, with one to eight chunks (B = 1, 8), and in several rounds."""
    p = problem(blocks + B, tuple(max(0, blocks * 64 - (b % 3)) for b in range(B)))
    out, lse, status = gpu_attention(in_table_of(p, 300))
    assert status == 0
    ref, rlse = oracle.attention(oracle.Geometry.of(p), p.k_cache, p.v_cache, p.q, p.k_tree, p.v_tree, p.scale)
    check_attention(out, ref, f"blocks={blocks} B={B}")
    np.testing.assert_allclose(lse, rlse, rtol=2e-3, atol=2e-3)


@pytest.mark.parametrize("lens,T", [((900, 333, 1000), 19), ((130, 64), 40), (tuple(range(500, 200, -5)), 40),
                                    (tuple(range(2600, 2400, -5)), 19)])
def test_attention_and_acceptance_back_to_back(lens, T):
    """Attention, acceptance that rewrites the lengths, attention, ...: launches that may all begin while the ones
    ahead of them still run.  One round of CTAs, and several (dispatched by length) through both kernels."""
    long = problem(11, lens, T=T)
    short = copy.copy(long)
    short.len = (long.len // 3).astype(np.int32)
    refs = [gpu_attention(x)[:2] for x in (long, short)]
    bt, srcs, st = sd.Batch.of(long), [sd.Batch.of(x) for x in (long, short)], sd.new_status()
    for s in srcs:
        s.len -= 1                                        # one node accepted: the lengths of long and short
    sd.sd_tree_prepare(bt, st)
    i32 = lambda *shape: torch.zeros(shape, dtype=torch.int32, device="cuda")
    draft, argmax, n_acc, path, tok = i32(bt.B, T) + 1, i32(bt.B * T), i32(bt.B), i32(bt.B, T), i32(bt.B, T)
    cache = sd.kv_layer(to_device(long.k_cache), to_device(long.v_cache))
    q, kt, vt = to_device(long.q), to_device(long.k_tree), to_device(long.v_tree)
    ws = torch.empty(sd.sd_workspace_bytes(bt), dtype=torch.uint8, device="cuda")
    runs = 16
    outs = torch.full((runs, bt.B, T, bt.Hq, bt.D), 7.0, dtype=torch.bfloat16, device="cuda")
    lses = torch.zeros((runs, bt.B, T, bt.Hq), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    for i in range(runs):
        sd.sd_accept_tree(srcs[i % 2], draft, argmax, n_acc, path, tok, bt.len, st)
        sd.sd_verify_attention(bt, cache, q, kt, vt, float(long.scale), outs[i], lses[i], ws, st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    for i in range(runs):
        np.testing.assert_array_equal(outs[i].float().cpu().numpy(), refs[i % 2][0])
        np.testing.assert_array_equal(lses[i].cpu().numpy(), refs[i % 2][1])
