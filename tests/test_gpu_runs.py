"""The SSD kernel for long runs of tiles at its edges: six tiles (the fewest it takes) and one more token, odd head
counts, two groups, leading tiles, segments, given states; heads that decay too fast for one reference per tile
(more than 2^-188 over its 128 tokens), and for products of factors at all (2^-96 over 32)."""
import math

import pytest
import torch

from paper_2603_06938_b200 import synth

import helpers as hp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,H,G,fast", [(25, 768, 5, 1, False), (38, 769, 4, 2, True), (25, 769, 6, 1, True),
                                          (13, 1537, 17, 1, True), (1, 5000, 12, 2, True), (76, 768, 4, 1, False)])
def test_long_runs_match_oracle(B, L, H, G, fast):
    cfg = synth.LayerConfig("runs", "bf16", B, L, 32, H, 64, 128, G, 4, 2, 128, h0_std=0.2)
    inp = synth.make_inputs(cfg, seed=60 + H)
    if fast:
        # log2 decay over n tokens: 16 step n / ln 2 -- 250 a tile, 63 a block for the first head, 110 a block (+- a
        # few) for the last one
        for head, step in ((0, 0.085), (H - 1, 0.149)):
            inp["A"][head] = -16.0
            inp["dt_bias"][head] = math.log(math.expm1(step))
        inp["dt"] *= 0.1
    got = hp.gpu_forward(cfg, inp)
    hp.compare_forward(cfg, inp, got, *hp.tolerances(cfg))


def test_vanishing_steps_in_front_of_fast_tokens():
    """Eight tokens of step size 0 lead every 32-token block of two heads, the others decay by 2^-99 in all: of one
    warp's rows some have decayed by nothing, some by more than 2^-96."""
    B, L, H = 25, 769, 6
    cfg = synth.LayerConfig("runs", "bf16", B, L, 32, H, 64, 128, 1, 4, 2, 128, h0_std=0.2)
    inp = synth.make_inputs(cfg, seed=70)
    for head in (0, H - 1):
        inp["A"][head] = -16.0
        inp["dt_bias"][head] = math.log(math.expm1(0.179))
        inp["dt"][..., head] = 0.0
        inp["dt"][:, torch.arange(L) % 32 < 8, head] = -200.0
    got = hp.gpu_forward(cfg, inp)
    hp.compare_forward(cfg, inp, got, *hp.tolerances(cfg))
