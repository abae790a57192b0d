"""GPU: the sampled tail where its split over a cluster of eight CTAs has its edges: trees of one node per warp and of
few, layers for one CTA, for every copying one and more than each copies while the draw goes on, a vocabulary that ends inside
a group of 32, rows of one round of loads and of several."""
import pytest

from test_gpu_sampled import test_fused_sampled_tail_equals_the_separate_calls_and_the_reference as compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,depth,L,V,Hd", [(64, 6, 1, 4096, 64), (9, 3, 7, 4097, 128), (33, 5, 8, 2049, 256), (60, 6, 29, 3000, 64),
                                            (17, 4, 36, 1025, 3584)])
def test_split_over_the_cluster(T, depth, L, V, Hd):
    compare("c5", dict(B=6, T=T, depth=depth, L=L, V=V, Hd=Hd, prefix=70), 3.0)
