"""GPU: draft-side aggregation where a CTA's ring of tiles wraps (more tasks than slots, separate and shared K and
V), where it just does not, and consecutive calls whose ends overlap."""
import numpy as np
import pytest
import torch

from oracle.draft_attention import feature_attention
from paper_2509_18824_b200 import binding as sd
from paper_2509_18824_b200 import workloads as wl
from paper_2509_18824_b200.step import to_device

pytestmark = pytest.mark.gpu


# tasks per SM on 148 SMs: 5, 12, 13, 25 and 49 (slots: 12 for separate K and V, 24 for one buffer)
@pytest.mark.parametrize("S,L,Q,H", [(367, 3, 1, 2), (444, 9, 5, 4), (445, 32, 8, 4), (917, 17, 2, 4), (1800, 28, 4, 4)])
@pytest.mark.parametrize("same", [False, True])
def test_ring_wraps(S, L, Q, H, same):
    g = np.random.default_rng(S + L)
    D = H * 128
    bf = lambda a: wl.f32_to_bf16_bits(a.astype(np.float32))
    qp, k = bf(g.standard_normal((Q, D)) * 4), bf(g.standard_normal((S, L, D)))
    v = k if same else bf(g.standard_normal((S, L, D)))
    qd, kd = to_device(qp), to_device(k)
    vd = kd if same else to_device(v)
    scale = 1.0 / np.sqrt(128)
    outs = [torch.full((S, Q, D), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(3)]
    for o in outs:
        sd.sd_draft_feature_attention(qd, kd, vd, H, scale, o)
    torch.cuda.synchronize()
    ref = feature_attention(wl.bf16_bits_to_f64(qp), wl.bf16_bits_to_f64(k), wl.bf16_bits_to_f64(v), H, scale)
    for o in outs:
        got = o.float().cpu().numpy()
        assert np.linalg.norm(got - ref) <= 5e-3 * np.linalg.norm(ref)
        per_row = np.linalg.norm((got - ref).reshape(S * Q * H, 128), axis=1) / np.linalg.norm(ref.reshape(S * Q * H, 128), axis=1)
        assert per_row.max() <= 3e-2
