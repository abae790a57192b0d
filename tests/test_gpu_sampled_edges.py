"""GPU: acceptance of drafts sampled from q where a thread's share of the vocabulary has its edges: fewer entries than
CTAs, one entry per thread and one more, slices that end inside a warp, and the largest vocabulary that a cluster
holds; chains one entry beyond it take the kernels that read the logits in passes."""
import numpy as np
import pytest

import oracle
from oracle import sampling as smp
from paper_2509_18824_b200 import workloads as wl
from test_gpu_sampled import (decisive_chain_inputs, decisive_tree_inputs, drafted_chain, drafted_tree, run_chain_q,
                              run_tree_q)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,T", [(1, 4), (7, 64), (4096, 64), (4097, 17), (12311, 64), (163840, 9)])
def test_tree_vocabulary_edges(V, T):
    w = wl.make("c5", attention=False, hidden_gain=24.0, B=2, T=T, depth=min(6, T - 2), L=1, V=V, Hd=64, prefix=70)
    lg = oracle.logits(w.hidden, w.W)
    inv_temp = 2.0
    q, tok = drafted_tree(w, lg, inv_temp, 0.5, V)
    u, wv, ref_n, ref_path, ref_out, _ = decisive_tree_inputs(w, tok, q, lg, inv_temp, np.random.default_rng(V + 1))
    n_acc, path, out_tok, new_len, status = run_tree_q(w, tok, q, inv_temp, u, wv)
    assert status == 0
    np.testing.assert_array_equal(n_acc, ref_n)
    np.testing.assert_array_equal(path, ref_path)
    np.testing.assert_array_equal(out_tok, ref_out)
    np.testing.assert_array_equal(new_len, w.len + ref_n)


@pytest.mark.parametrize("V,T", [(1, 2), (7, 64), (4096, 11), (4097, 11), (163840, 5), (163841, 5)])
@pytest.mark.parametrize("spread", [0.02, 1.0])                  # a drafter close to the target, one far from it
def test_chain_vocabulary_edges(V, T, spread):
    w = wl.make("chain11", attention=False, hidden_gain=24.0, B=2, T=T, L=1, V=V, Hd=64, prefix=70)
    lg = oracle.logits(w.hidden, w.W)
    inv_temp = 2.0
    q, tok, q_tok = drafted_chain(w, lg, inv_temp, spread, V)
    p, _ = smp.softmax_rows(lg, inv_temp)
    u, wv, ref_n, ref_out = decisive_chain_inputs(w, tok, q, lambda r: p[r], np.random.default_rng(V + 1))
    n_acc, path, out_tok, new_len, status = run_chain_q(w, tok, q, q_tok, inv_temp, u, wv, keep_logits=True)
    assert status == 0
    np.testing.assert_array_equal(n_acc, ref_n)
    np.testing.assert_array_equal(out_tok, ref_out)
    np.testing.assert_array_equal(new_len, w.len + ref_n)
    for b in range(2):
        np.testing.assert_array_equal(path[b, :ref_n[b]], np.arange(ref_n[b]))
