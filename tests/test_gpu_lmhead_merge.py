"""GPU: the merges of the LM head's per-CTA candidates and soft-max partials: the candidates of 1, 2, 8, 10 and of all
SMs' CTAs (a pair of CTAs from 129 vocabulary rows on: their number is even), rows that fill the merging CTAs' 8 and 64
rows and one more or less."""
import pytest

from test_gpu_lmhead_pieces import test_pieces as compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [1, 128, 129, 1024, 1025, 18944, 19201])
@pytest.mark.parametrize("M", [1, 8, 63, 64, 65, 130])
def test_rows_and_candidates(M, V):
    compare(M, 64, V)
