"""The recurrence cut over the SMs: sequences in 8, 9, 17 and 18 segments (the scan keeps eight in flight)
and batches whose leading tiles go to a second set of blocks (one, two and four of them, odd head counts,
ragged last tiles), against the oracle."""
import pytest

from paper_2603_06938_b200 import synth

import helpers as hp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,H", [(1, 1000, 8), (1, 1025, 3), (2, 2049, 2), (1, 2177, 6),        # segments
                                   (5, 513, 31), (25, 641, 6), (9, 1537, 17)])                    # leading tiles
def test_split_sequences_match_oracle(B, L, H):
    cfg = synth.LayerConfig("splits", "bf16", B, L, 32, H, 64, 128, 1, 4, 2, 128, h0_std=0.2)
    inp = synth.make_inputs(cfg, seed=90 + H)
    got = hp.gpu_forward(cfg, inp)
    hp.compare_forward(cfg, inp, got, *hp.tolerances(cfg))
