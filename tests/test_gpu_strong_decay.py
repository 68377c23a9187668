"""Heads that decay by far more than fp32's smallest number inside one 32-token block: a token's own term, and those of
the few tokens in front of it, stay whatever the rest of the block decays by.  No skip term, so that y is the
readout alone; the first three heads decay by 2^-140, 2^-200 and 2^-400 a block, in some cases with blocks in between
that hardly decay."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2603_06938_b200 import synth

import helpers as hp
import test_gpu_backward as tb
import test_gpu_packed as tp

pytestmark = pytest.mark.gpu


def strong_inputs(cfg, seed, slow_blocks):
    inp = synth.make_inputs(cfg, seed=seed)
    inp["D"] = None
    slow = (torch.arange(cfg.L) // 32) % 4 == 2
    for head, bits in zip(range(cfg.H), (140, 200, 400)):
        inp["A"][head] = -16.0
        inp["dt_bias"][head] = math.log(math.expm1(bits * math.log(2.0) / (16 * 32)))
        inp["dt"][..., head] *= 0.1
        if slow_blocks:
            inp["dt"][:, slow, head] = -7.0
    return inp


# the tile kernel: one partial tile, several tiles, segments; the kernel for six tiles and more: one segment,
# leading tiles; the CUDA cores
@pytest.mark.parametrize("dtype,B,L,H,slow", [("bf16", 2, 70, 3, False), ("bf16", 2, 300, 4, True), ("bf16", 1, 1025, 3, False),
                                              ("bf16", 25, 769, 6, False), ("bf16", 25, 769, 6, True),
                                              ("bf16", 50, 800, 3, True), ("fp32", 2, 300, 3, True)])
def test_forward(dtype, B, L, H, slow):
    cfg = synth.LayerConfig("strong", dtype, B, L, 32, H, 64, 128, 1, 4, 2, 128, h0_std=0.2)
    inp = strong_inputs(cfg, 80 + H, slow)
    got = hp.gpu_forward(cfg, inp)
    hp.compare_forward(cfg, inp, got, *hp.tolerances(cfg))


def test_packed():
    lens = [300, 2, 129]
    cfg = synth.LayerConfig("strong", "bf16", 1, sum(lens), 128, 3, 64, 128, 1, 4, 2, 64)
    inp = strong_inputs(cfg, 85, True)
    tp.check_packed(cfg, inp, lens, tp.packed_forward(cfg, inp, lens))


@pytest.mark.parametrize("B,L,H,slow", [(2, 128, 3, False), (1, 300, 3, True)])
def test_weight_gradients(B, L, H, slow):
    cfg = tb.cfg_of(B=B, L=L, H=H, h0_std=0.3)
    inp = strong_inputs(cfg, 86, slow)
    gen = torch.Generator().manual_seed(87)
    dy = torch.randn(B, L, H, cfg.P, generator=gen).to(torch.bfloat16)
    dWr, dWe, idx = tb.gpu_backward(cfg, inp, dy, h0=inp["h0"])
    ref = oracle.backward_weights(synth.f64(inp["u"]), synth.f64(inp["x"]), synth.f64(inp["dt"]), synth.f64(inp["W_r"]),
                                  synth.f64(inp["W_e"]), synth.f64(inp["A"]), synth.f64(inp["dt_bias"]), synth.f64(dy),
                                  cfg.k, G=1, h0=synth.f64(inp["h0"]), forced_idx=idx.numpy())
    assert tb.rel_per_expert(dWe.numpy(), ref["dW_e"]) <= 2e-2
    assert hp.max_rel(dWr.double().numpy(), np.asarray(ref["dW_r"])) <= 2e-2
