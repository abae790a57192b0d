"""A bounded wait that runs out: the kernels give up, report SD_ERR_TIMEOUT through the status word and
return normally, and the next ordinary call on the same stream is correct.

The waits are made to run out from the host side only, through the library's test hooks (environment
variables read at every launch): SDV_TEST_WAIT_CYCLES shortens the bound of every barrier wait to about a
tenth of a millisecond, SDV_TEST_WITHHOLD=1 makes one role skip a single arrival (the softmax warps never
report their first tile / the MMA thread never reports its first accumulator), so that its consumer waits
for something that does not come.  Nothing faults, traps or spins without a bound.
"""
import numpy as np
import pytest
import torch

import oracle
from oracle import sampling as smp
from oracle.draft_attention import feature_attention
from paper_2509_18824_b200 import binding as sd
from paper_2509_18824_b200 import workloads as wl
from gpu_util import gpu_attention, check_attention, gpu_lmhead, check_argmax
from paper_2509_18824_b200.step import to_device
from test_gpu_attention_tiles import problem
from test_gpu_sampled import (decisive_chain_inputs, decisive_tree_inputs, drafted_chain, drafted_tree, run_chain_q,
                              run_tree_q)

pytestmark = pytest.mark.gpu


def with_short_waits(monkeypatch, fn):
    """fn with the hooks set around it only (the calls in front of it are ordinary ones)."""
    def call(*args, **kw):
        with monkeypatch.context() as m:
            m.setenv("SDV_TEST_WAIT_CYCLES", "200000")
            m.setenv("SDV_TEST_WITHHOLD", "1")
            fn(*args, **kw)
    return call


def test_attention_wait_runs_out_and_the_next_call_is_fine(monkeypatch):
    w = wl.make("c1", lmhead=False, q_gain=45.0)                 # one sequence, one KV head, 32 rows: one CTA
    ref, _ = oracle.attention(oracle.Geometry.of(w), w.k_cache[0], w.v_cache[0], w.q[0], w.k_tree[0],
                              w.v_tree[0], w.scale)
    monkeypatch.setenv("SDV_TEST_CHUNKS", "1")                   # no key chunks: no cluster
    monkeypatch.setenv("SDV_TEST_WAIT_CYCLES", "200000")
    monkeypatch.setenv("SDV_TEST_WITHHOLD", "1")
    out, lse, status = gpu_attention(w, layer=0)                 # returns: the call and the synchronisation after it
    assert status == sd.SD_ERR_TIMEOUT
    monkeypatch.delenv("SDV_TEST_WITHHOLD")
    monkeypatch.delenv("SDV_TEST_WAIT_CYCLES")
    for _ in range(2):                                           # the context is intact: ordinary calls, right results
        out, lse, status = gpu_attention(w, layer=0)
        assert status == 0
        check_attention(out, ref, "after a timed-out call")


def all_layers(p, layers):
    """`layers` times the same layer in one call: (first and last output, status)."""
    bt, st = sd.Batch.of(p), sd.new_status()
    sd.sd_tree_prepare(bt, st)
    kc, vc, q, kt, vt = (to_device(x) for x in (p.k_cache, p.v_cache, p.q, p.k_tree, p.v_tree))
    o = [torch.full((p.B, p.T_max, p.Hq, p.D), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(layers)]
    ws = torch.empty(sd.sd_workspace_bytes(bt), dtype=torch.uint8, device="cuda")
    same = lambda x: [x] * layers
    sd.sd_verify_attention_layers(bt, sd.AttentionLayerSet(same(kc), same(vc), same(q), same(kt), same(vt), o), float(p.scale), ws, st)
    torch.cuda.synchronize()
    return [x.float().cpu().numpy() for x in (o[0], o[-1])], int(st.item())


# key chunks in clusters: the 128-key kernel, and (32 layers of short sequences) the 64-key one, whole and in chunks
@pytest.mark.parametrize("lens,layers,chunks", [((700, 2300), 1, 2), ((700, 2300), 1, 3), ((700, 2300), 1, 8),
                                                ((900, 333, 1000), 32, 1), ((900, 333, 1000), 32, 2)])
def test_attention_in_chunks_wait_runs_out_and_the_next_call_is_fine(monkeypatch, lens, layers, chunks):
    p = problem(sum(lens), lens, T=12, Hq=8, Hkv=2, gain=1.0)
    ref, _ = oracle.attention(oracle.Geometry.of(p), p.k_cache, p.v_cache, p.q, p.k_tree, p.v_tree, p.scale)
    monkeypatch.setenv("SDV_TEST_CHUNKS", str(chunks))
    with monkeypatch.context() as m:
        m.setattr(sd, "sd_verify_attention_layers", with_short_waits(m, sd.sd_verify_attention_layers))
        assert all_layers(p, layers)[1] == sd.SD_ERR_TIMEOUT
    for _ in range(2):
        outs, status = all_layers(p, layers)
        assert status == 0
        for out in outs:
            check_attention(out, ref, "after a timed-out call")


def test_lmhead_wait_runs_out_and_the_next_call_is_fine(monkeypatch):
    g = np.random.default_rng(1)
    M, Hd, V = 8, 128, 100                                       # at most 128 vocabulary rows: the single-CTA kernel
    h = wl.f32_to_bf16_bits(g.standard_normal((M, Hd)).astype(np.float32))
    W = wl.f32_to_bf16_bits((g.standard_normal((V, Hd)) / np.sqrt(Hd)).astype(np.float32))
    hd, Wd = to_device(h), to_device(W)
    am = torch.full((M,), -5, dtype=torch.int32, device="cuda")
    ws = torch.empty(sd.sd_workspace_bytes(None, M, V), dtype=torch.uint8, device="cuda")
    st = sd.new_status()
    monkeypatch.setenv("SDV_TEST_WAIT_CYCLES", "200000")
    monkeypatch.setenv("SDV_TEST_WITHHOLD", "1")
    sd.sd_lmhead_argmax(hd, Wd, am, None, ws, st)
    torch.cuda.synchronize()
    assert int(st.item()) == sd.SD_ERR_TIMEOUT
    monkeypatch.delenv("SDV_TEST_WITHHOLD")
    monkeypatch.delenv("SDV_TEST_WAIT_CYCLES")
    am2, mx2 = gpu_lmhead(h, W)
    ram, t1, t2 = oracle.lmhead(h, W)
    check_argmax(am2, mx2, ram, t1, t2)


# one pair of CTAs, pairs with one and several tiles, two MMAs a step (one accumulator), leftover tiles cut into pieces, two row
# blocks in a launch, and a third one behind them
@pytest.mark.parametrize("M,V", [(8, 200), (60, 4099), (60, 60000), (300, 4099), (480, 25000), (700, 4099), (1100, 25000)])
def test_lmhead_pair_wait_runs_out_and_the_next_call_is_fine(monkeypatch, M, V):
    g = np.random.default_rng(M)
    Hd = 128
    h = wl.f32_to_bf16_bits(g.standard_normal((M, Hd)).astype(np.float32))
    W = wl.f32_to_bf16_bits((g.standard_normal((V, Hd)) / np.sqrt(Hd)).astype(np.float32))
    hd, Wd = to_device(h), to_device(W)
    am = torch.full((M,), -5, dtype=torch.int32, device="cuda")
    ws = torch.empty(sd.sd_workspace_bytes(None, M, V), dtype=torch.uint8, device="cuda")
    st = sd.new_status()
    with_short_waits(monkeypatch, sd.sd_lmhead_argmax)(hd, Wd, am, None, ws, st)
    torch.cuda.synchronize()
    assert int(st.item()) == sd.SD_ERR_TIMEOUT
    am2, mx2 = gpu_lmhead(h, W)
    ram, t1, t2 = oracle.lmhead(h, W)
    check_argmax(am2, mx2, ram, t1, t2)


# one task, one per CTA, two per CTA, and thirteen: more than a CTA's ring of separate K and V tiles holds
@pytest.mark.parametrize("S,L,H", [(1, 28, 1), (18, 3, 8), (37, 32, 8), (481, 5, 4)])
@pytest.mark.parametrize("same", [False, True])
def test_draft_wait_runs_out_and_the_next_call_is_fine(monkeypatch, S, L, H, same):
    g = np.random.default_rng(S)
    Q, D, scale = 4, H * 128, 1.0 / np.sqrt(128)
    bf = lambda *shape: wl.f32_to_bf16_bits(g.standard_normal(shape).astype(np.float32))
    qp, k = bf(Q, D), bf(S, L, D)
    v = k if same else bf(S, L, D)
    qd, kd = to_device(qp), to_device(k)
    vd = kd if same else to_device(v)
    out = torch.full((S, Q, D), 7.0, dtype=torch.bfloat16, device="cuda")

    def rows():
        sd.sd_draft_feature_attention(qd, kd, vd, H, scale, out)
        torch.cuda.synchronize()
        return out.float().cpu().numpy()

    ref = feature_attention(wl.bf16_bits_to_f64(qp), wl.bf16_bits_to_f64(k), wl.bf16_bits_to_f64(v), H, scale)
    monkeypatch.setenv("SDV_TEST_WAIT_CYCLES", "200000")
    monkeypatch.setenv("SDV_TEST_WITHHOLD", "1")
    assert np.isnan(rows()).all()                                # (every copy waits for bytes that do not come)
    monkeypatch.delenv("SDV_TEST_WITHHOLD")
    monkeypatch.delenv("SDV_TEST_WAIT_CYCLES")
    for _ in range(2):
        got = rows()
        assert np.linalg.norm(got - ref) <= 5e-3 * np.linalg.norm(ref)


@pytest.mark.parametrize("cfg,over", [("c1", dict(V=1000, Hd=64)), ("c4", dict(L=1, V=4099, Hd=64, prefix_range=(40, 300)))])
def test_sampled_tree_wait_runs_out_and_the_next_call_is_fine(monkeypatch, cfg, over):
    """One CTA of each cluster keeps its sums to itself: the others' exchange runs out."""
    w = wl.make(cfg, attention=False, hidden_gain=24.0, **over)
    lg = oracle.logits(w.hidden, w.W)
    q, tok = drafted_tree(w, lg, 2.0, 0.8, 3)
    u, wv, ref_n, ref_path, ref_out, _ = decisive_tree_inputs(w, tok, q, lg, 2.0, np.random.default_rng(4))
    with monkeypatch.context() as m:
        m.setattr(sd, "sd_accept_tree_sampled_q", with_short_waits(m, sd.sd_accept_tree_sampled_q))
        assert run_tree_q(w, tok, q, 2.0, u, wv)[-1] == sd.SD_ERR_TIMEOUT
    n_acc, path, out_tok, _, status = run_tree_q(w, tok, q, 2.0, u, wv)
    assert status == 0
    for got, ref in ((n_acc, ref_n), (path, ref_path), (out_tok, ref_out)):
        np.testing.assert_array_equal(got, ref)


@pytest.mark.parametrize("B", [1, 16])
def test_sampled_chain_wait_runs_out_and_the_next_call_is_fine(monkeypatch, B):
    w = wl.make("chain11", attention=False, hidden_gain=24.0, L=1, V=3000, Hd=128, prefix=70, B=B)
    lg = oracle.logits(w.hidden, w.W)
    q, tok, q_tok = drafted_chain(w, lg, 2.5, 0.6, 3)
    p, _ = smp.softmax_rows(lg, 2.5)
    u, wv, ref_n, ref_out = decisive_chain_inputs(w, tok, q, lambda r: p[r], np.random.default_rng(4))
    with monkeypatch.context() as m:
        m.setattr(sd, "sd_accept_chain_sampled", with_short_waits(m, sd.sd_accept_chain_sampled))
        assert run_chain_q(w, tok, q, q_tok, 2.5, u, wv, keep_logits=True)[-1] == sd.SD_ERR_TIMEOUT
    n_acc, _, out_tok, _, status = run_chain_q(w, tok, q, q_tok, 2.5, u, wv, keep_logits=True)
    assert status == 0
    np.testing.assert_array_equal(n_acc, ref_n)
    np.testing.assert_array_equal(out_tok, ref_out)
