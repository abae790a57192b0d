"""GPU: LM head above 512 rows, where two row blocks share a launch: a last block that is narrower, an odd number of blocks,
whole tiles alone, tiles cut into pieces, fewer tiles than pairs; arg-max, statistics with and without it, group statistics, kept
logits and the probabilities of more than 512 stop rows."""
import copy

import numpy as np
import pytest
import torch

import oracle
from oracle import sampling as smp
from paper_2509_18824_b200 import binding as sd
from paper_2509_18824_b200 import workloads as wl
from paper_2509_18824_b200.step import to_device
from gpu_util import check_argmax, gpu_lmhead
from test_gpu_sampled import good_drafts, run_sampled

pytestmark = pytest.mark.gpu


# 256-row tiles: 2, 9, 37 (as many as the pairs of a block on 148 SMs), 75, 38 and 150
@pytest.mark.parametrize("M,Hd,V", [(513, 128, 257), (1024, 64, 2049), (961, 192, 9472), (1025, 64, 19000), (1537, 64, 9500), (700, 64, 38300)])
def test_row_blocks(M, Hd, V):
    g = np.random.default_rng(M + V)
    h = wl.f32_to_bf16_bits((g.standard_normal((M, Hd)) * 3).astype(np.float32))
    W = wl.f32_to_bf16_bits((g.standard_normal((V, Hd)) / np.sqrt(Hd)).astype(np.float32))
    ref, t1, t2 = oracle.lmhead(h, W)
    check_argmax(*gpu_lmhead(h, W), ref, t1, t2)
    inv_temp = 1.25
    am = torch.full((M,), -5, dtype=torch.int32, device="cuda")
    mx, lse = torch.zeros(M, device="cuda"), torch.zeros(M, device="cuda")
    kept = torch.full((M, V), float("nan"), device="cuda")
    ws = torch.empty(sd.sd_workspace_bytes(None, M, V), dtype=torch.uint8, device="cuda")
    st = sd.new_status()
    sd.sd_lmhead_stats_logits(to_device(h), to_device(W), inv_temp, am, mx, lse, kept, ws, st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    check_argmax(am.cpu().numpy(), mx.cpu().numpy(), ref, t1, t2)
    logits = oracle.logits(h, W)
    # Hd products of bf16, added up in fp32: at most Hd 2^-24 of the sum of their magnitudes
    bound = Hd * 2.0 ** -24 * (np.abs(wl.bf16_bits_to_f32(h)) @ np.abs(wl.bf16_bits_to_f32(W)).T)
    assert (np.abs(kept.cpu().numpy() - logits) <= bound + 1e-6).all()
    _, rlse = smp.softmax_rows(logits, inv_temp)
    np.testing.assert_allclose(lse.cpu().numpy(), rlse, rtol=0, atol=3e-4)


# row blocks of 272 and 241 rows, the latter with fewer columns of its own; of 368, 368 and 364: two side by side, then one
@pytest.mark.parametrize("M,rows", [(513, 272), (1100, 368)])
def test_row_blocks_and_calls_for_each(M, rows):
    """The same bits as calls for the rows of each block alone."""
    V, Hd = 128256, 2048
    g = torch.Generator(device="cuda").manual_seed(M)
    h = torch.randn((M, Hd), device="cuda", generator=g).to(torch.bfloat16)
    W = torch.randn((V, Hd), device="cuda", generator=g).to(torch.bfloat16)
    ws = torch.empty(sd.sd_workspace_bytes(None, M, V), dtype=torch.uint8, device="cuda")
    st = sd.new_status()

    def call(x):
        n = x.shape[0]
        am = torch.full((n,), -5, dtype=torch.int32, device="cuda")
        mx, lse, kept = torch.zeros(n, device="cuda"), torch.zeros(n, device="cuda"), torch.full((n, V), float("nan"), device="cuda")
        sd.sd_lmhead_stats_logits(x, W, 1.0 / 32, am, mx, lse, kept, ws, st)
        am2 = torch.full((n,), -5, dtype=torch.int32, device="cuda")
        sd.sd_lmhead_argmax(x, W, am2, None, ws, st)
        assert torch.equal(am, am2)
        return am, mx, lse, kept

    whole = call(h)
    for r in range(0, M, rows):
        part = call(h[r:r + rows].contiguous())
        for k in (0, 1, 3):
            assert torch.equal(whole[k][r:r + rows], part[k])
        # (sums of V fp32 terms, brought together from other CTAs' parts: a few 2^-24 of the sum in each of some ten merges)
        assert (whole[2][r:r + rows] - part[2]).abs().max().item() <= 1e-5
    assert int(st.item()) == 0


@pytest.mark.parametrize("M,V", [(700, 2049), (1100, 4099), (513, 100)])       # (100: one CTA at a time, no pairs)
def test_group_statistics(M, V):
    """Maximum and sum of every 32 vocabulary rows, with an arg-max and without, over both blocks of a launch."""
    Hd, inv_temp = 64, 1.25
    g = np.random.default_rng(M)
    h = wl.f32_to_bf16_bits((g.standard_normal((M, Hd)) * 3).astype(np.float32))
    W = wl.f32_to_bf16_bits((g.standard_normal((V, Hd)) / np.sqrt(Hd)).astype(np.float32))
    hd, Wd = to_device(h), to_device(W)
    ws, st = torch.empty(sd.sd_workspace_bytes(None, M, V), dtype=torch.uint8, device="cuda"), sd.new_status()
    res = []
    for am in (torch.full((M,), -5, dtype=torch.int32, device="cuda"), None):
        lse, gs = torch.zeros(M, device="cuda"), torch.full(sd.group_stats_shape(M, V), float("nan"), device="cuda")
        sd.sd_lmhead_stats(hd, Wd, inv_temp, am, None, lse, ws, st, group_stats=gs)
        res.append((lse.cpu().numpy(), gs.cpu().numpy()))
    assert int(st.item()) == 0
    for a, b in zip(*res):
        np.testing.assert_array_equal(a, b)
    logits = oracle.logits(h, W)
    lse, gs = res[0]
    # Hd products of bf16, added up in fp32: at most Hd 2^-24 of the sum of their magnitudes
    bound = (Hd * 2.0 ** -24 * (np.abs(wl.bf16_bits_to_f32(h)) @ np.abs(wl.bf16_bits_to_f32(W)).T)).max() + 1e-6
    full = np.full((M, (V + 31) // 32 * 32), -np.inf)
    full[:, :V] = logits
    groups = full.reshape(M, -1, 32).transpose(1, 0, 2)
    assert np.abs(gs[..., 0] - groups.max(axis=2)).max() <= bound
    # the terms' exponents move by twice that, ex2.approx (2^-22) and 32 roundings of 2^-24 come on top
    ref = np.exp((groups - groups.max(axis=2, keepdims=True)) * inv_temp).sum(axis=2)
    np.testing.assert_allclose(gs[..., 1], ref, rtol=2 * bound * inv_temp + 2.0 ** -18)
    np.testing.assert_allclose(lse, smp.softmax_rows(logits, inv_temp)[1], rtol=0, atol=3e-4)


def test_probabilities_of_more_than_512_stop_rows():
    """600 sequences whose last tokens are drawn from a second pass over W: the tokens of three calls for 200 each."""
    w = wl.make("chain11", attention=False, hidden_gain=24.0, L=1, V=3000, Hd=128, prefix=70, B=600)
    T = w.T_max
    tok = good_drafts(w, oracle.logits(w.hidden, w.W), 1)
    g = np.random.default_rng(7)
    u, wv = g.random((600, T)).astype(np.float32), g.random(600).astype(np.float32)
    whole = run_sampled(w, tok, 2.5, u, wv, groups=False)
    assert whole[-1] == 0 and (whole[0] > 1).any()
    for b in range(0, 600, 200):
        x, some = copy.copy(w), slice(b, b + 200)
        x.B, x.hidden = 200, w.hidden[b * T:(b + 200) * T]
        for name in ("len", "n_nodes", "parents", "block_table"):
            setattr(x, name, np.ascontiguousarray(getattr(w, name)[some]))
        part = run_sampled(x, tok[some], 2.5, u[some], wv[some], groups=False)
        assert part[-1] == 0
        for all_of, here in zip(whole[:4], part[:4]):
            np.testing.assert_array_equal(all_of[some], here)
