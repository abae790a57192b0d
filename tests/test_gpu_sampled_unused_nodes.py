"""GPU: acceptance at a temperature where sequences use fewer nodes than their slots: whatever stands in the slots behind
them (parents, tokens outside the vocabulary, NaN uniforms and draft probabilities) must not matter, and is not reported."""
import numpy as np
import pytest
import torch

import oracle
from oracle import sampling as smp
from paper_2509_18824_b200 import workloads as wl
from paper_2509_18824_b200.step import VerifyStep, to_device
from test_gpu_sampled import (decisive_chain_inputs, decisive_tree_inputs, decisive_uniforms, drafted_chain, drafted_tree,
                              good_drafts, run_chain_q, run_sampled, run_tree_q, step_outputs)

pytestmark = pytest.mark.gpu
NODES = [1, 31, 32, 33, 64, 2]
JUNK_PARENTS = [-1, 63, 0, 1 << 30, -(1 << 31), 5]
JUNK_TOKENS = [-1, 1 << 30, 0, -(1 << 31), (1 << 31) - 1, 4099]


def ragged(cfg, **over):
    w = wl.make(cfg, hidden_gain=24.0, B=len(NODES), T=64, prefix=70, V=4099, Hd=128, **over)
    w.n_nodes = np.array(NODES, dtype=np.int32)
    return w


def junk(w, tok, *floats):
    """Junk in the unused slots of the parents, the tokens and the given float arrays."""
    w.parents = w.parents.copy()
    for b, n in enumerate(NODES):
        k = 64 - n
        w.parents[b, n:] = np.resize(JUNK_PARENTS, k)
        tok[b, n:] = np.resize(JUNK_TOKENS, k)
        for x in floats:
            x[b, n:] = np.nan


def test_top_k_tail():
    w = ragged("c5", depth=6, L=3)
    lg = oracle.logits(w.hidden, w.W)
    p64, lse64 = smp.softmax_rows(lg, 3.0)
    tok = good_drafts(w, lg, 5)
    g = np.random.default_rng(21)
    u, ref_n, ref_path, stop_R = decisive_uniforms(w, tok, lambda r: p64[r], g)
    wv = g.random(len(NODES)).astype(np.float32)
    clean = w.parents
    junk(w, tok, u)
    w.draft_tok = tok
    vs = VerifyStep(w)
    vs.tail_sampled(3.0, to_device(u), to_device(wv))
    torch.cuda.synchronize()
    vs.check_status()
    got = step_outputs(vs)
    apart = run_sampled(w, tok, 3.0, u, wv)
    assert apart[4] == 0
    for name, x in zip(("n_acc", "path", "out_tok", "new_len"), apart):
        np.testing.assert_array_equal(got[name], x, err_msg=name)
    np.testing.assert_allclose(got["lse"], lse64, rtol=0, atol=5e-4)
    np.testing.assert_array_equal(got["n_acc"], ref_n)
    np.testing.assert_array_equal(got["path"], ref_path)
    np.testing.assert_array_equal(got["new_len"], w.len + ref_n)
    close_calls = 0
    for b, n in enumerate(NODES):
        last = int(ref_path[b, ref_n[b] - 1])
        excl = [int(tok[b, c]) for c in smp.children_of(clean[b], n, last)]
        t_ref, margin = smp.residual_sample(p64[b * 64 + last], excl, float(stop_R[b]), float(wv[b]))
        t_got = int(got["out_tok"][b, ref_n[b] - 1])
        assert t_got not in excl and (t_got == t_ref or margin <= 2e-5 * max(float(stop_R[b]), 1e-3)), (b, t_got, t_ref, margin)
        close_calls += t_got != t_ref
    assert close_calls <= 1 and (ref_n > 1).any()
    G = oracle.Geometry.of(w)
    for l in range(w.L):
        rk, rv = w.k_cache[l].copy(), w.v_cache[l].copy()
        oracle.compact(G, rk, rv, w.k_tree[l], w.v_tree[l], ref_n, ref_path)
        np.testing.assert_array_equal(got["k"][l].view(np.uint16), rk)
        np.testing.assert_array_equal(got["v"][l].view(np.uint16), rv)


def test_sampled_tree():
    w = ragged("c5", attention=False, depth=6, L=1)
    lg = oracle.logits(w.hidden, w.W)
    q, tok = drafted_tree(w, lg, 2.0, 0.5, 13)
    u, wv, ref_n, ref_path, ref_out, _ = decisive_tree_inputs(w, tok, q, lg, 2.0, np.random.default_rng(14))
    junk(w, tok, u)
    n_acc, path, out_tok, new_len, status = run_tree_q(w, tok, q, 2.0, u, wv)
    assert status == 0 and (ref_n > 1).any()
    np.testing.assert_array_equal(n_acc, ref_n)
    np.testing.assert_array_equal(path, ref_path)
    np.testing.assert_array_equal(out_tok, ref_out)
    np.testing.assert_array_equal(new_len, w.len + ref_n)


@pytest.mark.parametrize("keep_logits", [True, False])
@pytest.mark.parametrize("spread", [0.02, 0.6])
def test_sampled_chain(spread, keep_logits):
    w = ragged("chain11", attention=False, L=1)
    lg = oracle.logits(w.hidden, w.W)
    p64, _ = smp.softmax_rows(lg, 2.0)
    q, tok, q_tok = drafted_chain(w, lg, 2.0, spread, 3)
    u, wv, ref_n, ref_out = decisive_chain_inputs(w, tok, q, lambda r: p64[r], np.random.default_rng(8))
    junk(w, tok, u, q_tok)
    n_acc, path, out_tok, new_len, status = run_chain_q(w, tok, q, q_tok, 2.0, u, wv, keep_logits)
    assert status == 0 and (ref_n > 1).any()
    np.testing.assert_array_equal(n_acc, ref_n)
    np.testing.assert_array_equal(out_tok, ref_out)
    np.testing.assert_array_equal(new_len, w.len + ref_n)
    for b in range(len(NODES)):
        assert list(path[b, :ref_n[b]]) == list(range(ref_n[b])) and (path[b, ref_n[b]:] == -1).all()


@pytest.mark.parametrize("keep_logits", [True, False])
def test_sampled_chain_accepted_to_its_end(keep_logits):
    w = ragged("chain11", attention=False, L=1)
    q, tok, q_tok = drafted_chain(w, oracle.logits(w.hidden, w.W), 2.0, 0.02, 3)
    u, wv = np.zeros((len(NODES), 64), np.float32), np.full(len(NODES), 0.5, np.float32)
    junk(w, tok, u, q_tok)
    n_acc, path, out_tok, new_len, status = run_chain_q(w, tok, q, q_tok, 2.0, u, wv, keep_logits)
    assert status == 0
    np.testing.assert_array_equal(n_acc, NODES)
    for b, n in enumerate(NODES):
        assert list(path[b]) == list(range(n)) + [-1] * (64 - n)
        assert list(out_tok[b, :n - 1]) == list(tok[b, 1:n]) and 0 <= out_tok[b, n - 1] < 4099 and (out_tok[b, n:] == -1).all()
