"""The streaming kernel's pairs of CTAs (H = 2048, more than 32 tokens) where groups of two tiles end: odd numbers of tiles,
a single tile, empty lists, several groups per pair."""
import pytest

from test_gpu_edges import step_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("I,T,L,B,density,clusters", [(330, 33, 2, 3, 0.9, 0), (64, 64, 2, 2, 0.4, 0), (700, 51, 3, 2, 0.8, 1),
                                                      (96, 51, 3, 4, 0.01, 0)])
def test_pairs_match_the_oracle(lib, I, T, L, B, density, clusters):
    step_case(lib, H=2048, I=I, T=T, L=L, B=B, density=density, variant=4, max_clusters=clusters, config=99)
