"""GPU: hidden states and weights with infinities and NaN: the fused tail at a temperature ends as the three calls that it stands for
(their outputs are no probabilities then, but the two must not part)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_18824_b200 import workloads as wl
from paper_2509_18824_b200.step import VerifyStep, to_device
from test_gpu_sampled import good_drafts, step_outputs

pytestmark = pytest.mark.gpu
INF, NINF, NAN = 0x7F80, 0xFF80, 0x7FC0                      # bf16 bit patterns


@pytest.mark.parametrize("seed", range(8))
@pytest.mark.parametrize("V,T,B", [(4099, 60, 8), (513, 20, 4)])
def test_fused_tail_equals_the_separate_calls(V, T, B, seed):
    w = wl.make("c5", hidden_gain=8.0, B=B, T=T, depth=4, L=2, V=V, Hd=128, prefix=70)
    w.draft_tok = good_drafts(w, oracle.logits(w.hidden, w.W), seed)
    g = np.random.default_rng(seed)
    w.hidden, w.W = w.hidden.copy(), w.W.copy()
    rows = g.permutation(B * T)[:B * T // 2]
    rows[:B // 2] = np.arange(B // 2) * T                     # some sequences' roots among them
    w.hidden[rows, g.integers(0, 128, rows.size)] = np.resize([INF, NINF, NAN, INF, NINF, 0x7F7F], rows.size)
    if seed >= 6:
        w.W[g.integers(0, V, 3), g.integers(0, 128, 3)] = [INF, NINF, NAN]
    u = g.random((B, T)).astype(np.float32)
    wv = g.random(B).astype(np.float32)
    res = []
    for fused in (False, True):
        vs = VerifyStep(w)
        vs.status.zero_()
        vs.tail_sampled(1.25, to_device(u), to_device(wv), fused=fused)
        torch.cuda.synchronize()
        res.append(dict(step_outputs(vs), status=int(vs.status.item())))
    assert res[0]["status"] == res[1]["status"]
    for key in ("lse", "n_acc", "path", "out_tok", "new_len"):
        np.testing.assert_array_equal(res[0][key], res[1][key], err_msg=key)
    for l in range(2):
        np.testing.assert_array_equal(res[0]["k"][l], res[1]["k"][l])
        np.testing.assert_array_equal(res[0]["v"][l], res[1]["v"][l])
