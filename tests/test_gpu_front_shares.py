"""The small front end with its tokens in shares (few experts, uneven shares, some of them without an entry) and
on both sides of the sizes where the grouped product takes over, against the oracle."""
import pytest

from paper_2603_06938_b200 import synth

import helpers as hp
import test_gpu_decode_front as front

pytestmark = pytest.mark.gpu


# shares; slots summed in the update and by their own kernel; sizes around the grouped product's (with 32 features
# the projection that takes over has fp32 streams as well, which the tolerance is for)
@pytest.mark.parametrize("B,F,H,P,N,E,k", [(256, 96, 1, 16, 16, 2, 2), (97, 64, 1, 16, 16, 2, 1), (50, 64, 1, 16, 16, 3, 2),
                                           (255, 64, 1, 16, 16, 1, 1), (130, 64, 3, 64, 128, 8, 8), (256, 64, 3, 64, 128, 16, 5),
                                           (160, 32, 1, 16, 16, 8, 8), (161, 32, 1, 16, 16, 8, 8)])
def test_decode_step(B, F, H, P, N, E, k):
    front.test_two_decode_steps_match_oracle(B, F, H, P, N, 1, E, k)


@pytest.mark.parametrize("T,F,E,k", [(95, 96, 2, 1), (96, 96, 2, 1), (127, 256, 2, 2), (128, 256, 2, 2), (256, 544, 3, 2),
                                     (200, 256, 4, 1)])
def test_short_forward(T, F, E, k):
    cfg = synth.LayerConfig("shares", "bf16", 1, T, F, 2, 64, 128, 1, E, k, 128)
    inp = synth.make_inputs(cfg, seed=20 + E)
    got = hp.gpu_forward(cfg, inp)
    hp.compare_forward(cfg, inp, got, *hp.tolerances(cfg))
