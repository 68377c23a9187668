"""The tensor-core adjoint at its edges: tile boundaries, walks cut into segments, head quads and shares of
odd head counts, two groups, a given initial state, decays beyond what a product of factors can hold."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_06938_b200 import synth

import helpers as hp
import test_gpu_backward as tb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,H,G,strong", [(1, 127, 1, 1, False), (2, 128, 5, 1, False), (1, 129, 4, 2, True),
                                            (1, 900, 3, 1, False), (1, 1409, 2, 2, True), (3, 257, 10, 2, False)])
def test_weight_gradients_at_the_edges_of_the_adjoint(B, L, H, G, strong):
    cfg = tb.cfg_of(B=B, L=L, H=H, G=G, h0_std=0.3)
    inp = synth.make_inputs(cfg, seed=600 + L)
    if strong:        # the last head halves 16 * 0.149 * 32 / ln 2 = 110 times per 32 tokens (+- a few): past the
        # 96 where exponents are formed entry by entry
        inp["A"] = -torch.linspace(4.0, 16.0, H)
        inp["dt_bias"] = torch.full((H,), float(np.log(np.expm1(0.149))))
        inp["dt"] = 0.1 * inp["dt"]
    gen = torch.Generator().manual_seed(601)
    dy = torch.randn(B, L, H, cfg.P, generator=gen).to(torch.bfloat16)
    dWr, dWe, idx = tb.gpu_backward(cfg, inp, dy, h0=inp["h0"])
    ref = oracle.backward_weights(synth.f64(inp["u"]), synth.f64(inp["x"]), synth.f64(inp["dt"]), synth.f64(inp["W_r"]),
                                  synth.f64(inp["W_e"]), synth.f64(inp["A"]), synth.f64(inp["dt_bias"]), synth.f64(dy),
                                  cfg.k, G=G, h0=synth.f64(inp["h0"]), forced_idx=idx.numpy())
    assert tb.rel_per_expert(dWe.numpy(), ref["dW_e"]) <= 2e-2
    assert hp.max_rel(dWr.double().numpy(), ref["dW_r"]) <= 2e-2
