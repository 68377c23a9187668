"""The small front end with its tokens in shares (few experts, uneven shares, some of them without an entry) and
on both sides of the sizes where the grouped product takes over, against the oracle."""
import pytest

from paper_2603_06938_b200 import synth

import helpers as hp
import test_gpu_decode_front as front

pytestmark = pytest.mark.gpu


# shares; slots summed in the update and by their own kernel; the grouped product's fp32 slots (one, two and more
# experts per token; wide streams) and the sizes next to them; few tokens without and with too many blocks to fuse
@pytest.mark.parametrize("B,F,H,P,N,G,E,k", [
    (256, 96, 1, 16, 16, 1, 2, 2), (97, 64, 1, 16, 16, 1, 2, 1), (50, 64, 1, 16, 16, 1, 3, 2), (255, 64, 1, 16, 16, 1, 1, 1),
    (130, 64, 3, 64, 128, 1, 8, 8), (256, 64, 3, 64, 128, 1, 16, 5), (256, 160, 3, 16, 128, 1, 16, 8),
    (64, 64, 4, 16, 128, 4, 5, 1), (9, 72 * 4, 4, 16, 128, 4, 16, 2), (200, 256, 8, 16, 64, 8, 6, 4),
    (3, 64, 8, 8, 128, 8, 16, 3), (4, 2048, 4, 16, 128, 4, 8, 2), (4, 2048, 4, 16, 128, 4, 10, 2)])
def test_decode_step(B, F, H, P, N, G, E, k):
    front.test_two_decode_steps_match_oracle(B, F, H, P, N, G, E, k)


@pytest.mark.parametrize("T,F,G,E,k", [(240, 96, 1, 8, 2), (241, 96, 1, 8, 2), (256, 544, 1, 3, 2), (200, 256, 1, 4, 1),
                                       (64, 64, 2, 2, 2), (63, 64, 4, 5, 1), (256, 2048, 4, 2, 1)])
def test_short_forward(T, F, G, E, k):
    cfg = synth.LayerConfig("shares", "bf16", 1, T, F, 2 * G, 64, 128, G, E, k, 128)
    inp = synth.make_inputs(cfg, seed=20 + E)
    got = hp.gpu_forward(cfg, inp)
    hp.compare_forward(cfg, inp, got, *hp.tolerances(cfg))
