"""The calls around the line between the products on CTA pairs and on narrow column tiles: many experts (most
tiles a few rows), short and long features, lists around half a tile, wide streams."""
import pytest

import test_gpu_pair_gemm as pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,F,G,N,E,k", [(1280, 1032, 1, 16, 64, 2), (1281, 1032, 1, 16, 64, 2), (7936, 64, 1, 128, 4, 1),
                                         (7937, 64, 1, 128, 4, 1), (1920, 1040, 1, 16, 16, 1), (1921, 1040, 1, 16, 16, 1),
                                         (1793, 2056, 1, 16, 16, 1), (520, 128, 8, 128, 8, 2), (24, 64, 8, 128, 64, 2)])
def test_projection_and_mix_match_oracle(T, F, G, N, E, k):
    pair.test_projection_and_mix_match_oracle(T, F, G, N, E, k)
