"""GPU: drafted tokens outside the vocabulary among the children of the node at which a walk stops: reported, and the other
sequence of the batch ends as without them, on every way to draw the last token."""
import numpy as np
import pytest
import torch

import oracle
from oracle import sampling as smp
from paper_2509_18824_b200 import binding as sd
from paper_2509_18824_b200 import workloads as wl
from paper_2509_18824_b200.step import VerifyStep, to_device
from test_gpu_sampled import good_drafts, run_sampled

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("way", ["fused", "groups", "second pass"])
@pytest.mark.parametrize("token", [-1, -33, -(1 << 31), 4099, 4128, 262144, (1 << 31) - 1])
def test_token_outside_the_vocabulary(token, way):
    w = wl.make("c5", attention=way == "fused", hidden_gain=24.0, B=2, T=17, depth=4, L=2, V=4099, Hd=128, prefix=70)
    u, wv = np.full((2, 17), 0.5, np.float32), np.full(2, 0.5, np.float32)
    kids = smp.children_of(w.parents[0], 17, 0)
    lg = oracle.logits(w.hidden, w.W)
    good = good_drafts(w, lg, 5)
    good[0, kids] = np.argsort(lg[0])[:len(kids)]             # sequence 0 stops at its root
    bad = good.copy()
    bad[0, kids[0]] = token
    got = []
    for tok in (good, bad):
        if way == "fused":
            w.draft_tok = tok
            vs = VerifyStep(w)
            vs.status.zero_()
            vs.tail_sampled(3.0, to_device(u), to_device(wv))
            torch.cuda.synchronize()
            out = [x.cpu().numpy() for x in (vs.n_acc, vs.path, vs.out_tok, vs.new_len)] + [int(vs.status.item())]
        else:
            out = run_sampled(w, tok, 3.0, u, wv, groups=way == "groups")
        got.append(out)
    assert got[0][4] == 0 and got[1][4] == sd.SD_ERR_BOUNDS
    for a, b in zip(got[0][:4], got[1][:4]):
        np.testing.assert_array_equal(a[1], b[1])
