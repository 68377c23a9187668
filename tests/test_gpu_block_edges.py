"""Convolution strips (16 tokens bf16, 8 fp32) and norm groups at their edges, through the block: calls
around a strip's length, every window width, a norm group longer than a thread block holds in registers."""
import pytest
import torch

from paper_2603_06938_b200 import synth

import helpers as hp
import test_gpu_block as tb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,L,H,G,d_conv", [("bf16", 15, 3, 1, 4), ("bf16", 16, 2, 2, 3), ("bf16", 17, 4, 2, 2),
                                                ("bf16", 2, 2, 1, 4), ("bf16", 1, 3, 1, 1), ("bf16", 33, 65, 1, 4),
                                                ("bf16", 600, 3, 1, 4), ("bf16", 530, 8, 2, 3),   # step sizes from the product's tail
                                                ("fp32", 8, 3, 3, 4), ("fp32", 9, 2, 1, 2)])
def test_block_edges_match_the_oracle_composition(dtype, L, H, G, d_conv):
    cfg = synth.LayerConfig("edges", dtype, 2, L, 64, H, 64, 128, G, 4, 2, 128)
    inp = synth.make_inputs(cfg, seed=700 + L)
    blk = tb.make_block(cfg, 800 + L, d_conv)
    gen = torch.Generator().manual_seed(9)
    cst = torch.randn(2, d_conv - 1, H * 64 + cfg.S, generator=gen).to(synth.torch_dtype(dtype)) if d_conv > 1 else None
    got = tb.gpu_block(cfg, inp, blk, inp["u"], conv_state=cst)
    ref = tb.oracle_block(cfg, inp, blk, inp["u"], got["idx"], conv_state=cst)
    bf16 = dtype == "bf16"
    # out: the tolerance of the block's other tests.  State: a handful of tokens do not average their
    # roundings, so x' (stored in bf16), x, the two slots of B' and B add up to at most five of 2^-8
    tol = dict(out=3e-2 if bf16 else 2e-4, conv_state=2.0 ** -7 if bf16 else 1e-5, h_final=5 * 2.0 ** -8 if bf16 else 1e-4)
    for name, t in tol.items():
        if got[name].numel():
            assert hp.max_rel(got[name].double().numpy(), ref[name]) <= t, name
