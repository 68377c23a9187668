"""The chunked CUDA-core recurrence (fp32, and bf16 shapes without a tensor-core kernel) at the edges of
its runs of 32 tokens, its clusters of up to eight CTAs and its padded channel rows, against the oracle."""
import pytest

from paper_2603_06938_b200 import synth

import helpers as hp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,L,P,N,G", [
    ("fp32", 1, 64, 16, 1), ("fp32", 31, 8, 16, 1), ("fp32", 32, 64, 48, 1), ("fp32", 33, 5, 16, 3),
    ("fp32", 256, 64, 16, 1), ("fp32", 257, 13, 32, 1), ("fp32", 289, 64, 256, 1), ("fp32", 520, 256, 16, 1),
    ("bf16", 65, 32, 64, 1), ("bf16", 300, 6, 32, 3)])
def test_chunked_recurrence_matches_oracle(dtype, L, P, N, G):
    cfg = synth.LayerConfig("chunk", dtype, 2, L, 64, 3, P, N, G, 4, 2, 64, h0_std=0.2)
    inp = synth.make_inputs(cfg, seed=300 + L)
    got = hp.gpu_forward(cfg, inp)
    # fp32: 1e-4 covers sums of up to 256 + 32 terms (each rounding 6e-8) with a wide margin
    hp.compare_forward(cfg, inp, got, *hp.tolerances(cfg))
