"""The chunked CUDA-core recurrence with as many sequences and heads as fill the SMs: clusters of four and two,
single blocks that carry the state over several runs, wide and narrow channel rows, with and without a given
state, against the oracle."""
import pytest

from paper_2603_06938_b200 import synth

import helpers as hp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,B,H,L,P,N,h0", [
    ("fp32", 5, 20, 150, 16, 16, 0.2), ("fp32", 10, 16, 97, 5, 16, 0.0), ("bf16", 8, 25, 70, 12, 32, 0.2),
    ("fp32", 20, 20, 65, 8, 16, 0.2), ("bf16", 20, 20, 33, 20, 48, 0.0), ("fp32", 20, 40, 40, 16, 16, 0.2),
    ("fp32", 3, 27, 75, 64, 256, 0.2), ("bf16", 4, 40, 34, 64, 256, 0.0), ("fp32", 5, 20, 9, 256, 64, 0.0)])
def test_many_heads_match_oracle(dtype, B, H, L, P, N, h0):
    cfg = synth.LayerConfig("fill", dtype, B, L, 32, H, P, N, 1, 4, 2, 64, h0_std=h0)
    inp = synth.make_inputs(cfg, seed=400 + L)
    got = hp.gpu_forward(cfg, inp)
    # fp32: 1e-4 covers sums of up to 256 + 32 terms (each rounding 6e-8) with a wide margin
    hp.compare_forward(cfg, inp, got, *hp.tolerances(cfg))
