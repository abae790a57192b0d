"""GPU: acceptance of drafts sampled from q around the vocabularies at which a thread's share grows from 8 to 16 and to 40
entries."""
import pytest

from test_gpu_sampled_edges import test_chain_vocabulary_edges as compare_chain
from test_gpu_sampled_edges import test_tree_vocabulary_edges as compare_tree

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [32761, 32768, 32769, 65536, 65537])
def test_share_of_a_thread(V):
    compare_tree(V, 9)
    compare_chain(V, 5, 1.0)
