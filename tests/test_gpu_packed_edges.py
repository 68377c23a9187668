"""Packed batches at the edges of their three ways through the SSD: sequences of one to four tokens
(stepped), one segment, several segments (whose first starts from the given state), in one batch."""
import pytest
import torch

from paper_2603_06938_b200 import synth

import test_gpu_packed as tp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens,G,h0", [([1, 2, 3, 4, 5], 1, True), ([4, 700, 1, 0, 129, 3], 2, True),
                                       ([2, 1300, 2], 1, False), ([512, 4, 513, 1025], 1, True)])
def test_stepped_and_tiled_sequences_in_one_batch(lens, G, h0):
    cfg = synth.LayerConfig("edges", "bf16", 1, sum(lens), 128, 3 * G, 64, 128, G, 4, 2, 64)
    inp = synth.make_inputs(cfg, seed=47)
    gen = torch.Generator().manual_seed(48)
    st = (0.1 * torch.randn(len(lens), cfg.H, cfg.P, cfg.N, generator=gen)).float() if h0 else None
    got = tp.packed_forward(cfg, inp, lens, h0=st)
    tp.check_packed(cfg, inp, lens, got, h0=st)
