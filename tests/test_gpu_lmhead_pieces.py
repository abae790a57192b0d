"""GPU: LM head above 256 rows where vocabulary tiles are cut into pieces along the hidden rows: fewer tiles than CTA
pairs, a few tiles beyond whole rounds, row counts whose last piece is narrower, several passes over the rows."""
import numpy as np
import pytest

import oracle
from paper_2509_18824_b200 import workloads as wl
from gpu_util import check_argmax, gpu_lmhead
from test_gpu_sampled import run_stats
from oracle import sampling as smp

pytestmark = pytest.mark.gpu


# 256-row tiles: 2, 9, 17 (fewer than 74 pairs), 75 and 150 (one and two beyond whole rounds on 148 SMs)
@pytest.mark.parametrize("M,Hd,V", [(257, 64, 511), (300, 192, 2300), (480, 128, 4099), (511, 64, 19000), (512, 64, 38300),
                                    (700, 64, 2049)])
def test_pieces(M, Hd, V):
    g = np.random.default_rng(M + V)
    h = wl.f32_to_bf16_bits((g.standard_normal((M, Hd)) * 3).astype(np.float32))
    W = wl.f32_to_bf16_bits((g.standard_normal((V, Hd)) / np.sqrt(Hd)).astype(np.float32))
    ref, t1, t2 = oracle.lmhead(h, W)
    check_argmax(*gpu_lmhead(h, W), ref, t1, t2)
    am, mx, lse = run_stats(h, W, 1.25)
    check_argmax(am, mx, ref, t1, t2)
    _, rlse = smp.softmax_rows(oracle.logits(h, W), 1.25)
    np.testing.assert_allclose(lse, rlse, rtol=0, atol=3e-4)
