"""GPU: LM head above 512 rows, where two row blocks share a launch: a last block that is narrower, an odd number of blocks,
whole tiles alone, tiles cut into pieces, fewer tiles than pairs; arg-max, statistics and kept logits."""
import numpy as np
import pytest
import torch

import oracle
from oracle import sampling as smp
from paper_2509_18824_b200 import binding as sd
from paper_2509_18824_b200 import workloads as wl
from paper_2509_18824_b200.step import to_device
from gpu_util import check_argmax, gpu_lmhead

pytestmark = pytest.mark.gpu


# 256-row tiles: 1, 9, 37 (as many as the pairs of a block on 148 SMs), 75 and 150
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
