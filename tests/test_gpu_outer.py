"""The expert-matrix gradient on CTA pairs at its edges: lists that start off a 16-byte boundary, lists
shorter and longer than a step of 64 entries, experts without tokens, tiles that end inside 256 columns,
every way a token can have slots; and the router's gradient over one and several groups of eight experts."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_06938_b200 import synth

import test_gpu_backward as tb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,F,N,G,E,k", [(1, 61, 64, 16, 1, 5, 1), (1, 203, 72, 64, 1, 64, 2), (3, 333, 328, 128, 1, 3, 2),
                                           (1, 515, 264, 128, 2, 9, 3), (2, 64, 512, 16, 1, 2, 2)])
def test_weight_gradients_at_the_edges_of_the_outer_products(B, L, F, N, G, E, k):
    P = 64 if N == 128 else 16
    cfg = tb.cfg_of(B=B, L=L, F=F, H=2 * G, P=P, N=N, G=G, E=E, k=k)
    inp = synth.make_inputs(cfg, seed=900 + L)
    gen = torch.Generator().manual_seed(901)
    dy = torch.randn(B, L, cfg.H, P, generator=gen).to(torch.bfloat16)
    dWr, dWe, idx = tb.gpu_backward(cfg, inp, dy, h0=None)
    ref = oracle.backward_weights(synth.f64(inp["u"]), synth.f64(inp["x"]), synth.f64(inp["dt"]), synth.f64(inp["W_r"]),
                                  synth.f64(inp["W_e"]), synth.f64(inp["A"]), synth.f64(inp["dt_bias"]), synth.f64(dy),
                                  k, G=G, forced_idx=idx.numpy())
    # the tolerance of the gradients' other tests; an expert with a handful of entries does not average their
    # roundings (mixed streams, slots, scaled rows: at most five of 2^-8), so its own scale is floored by a
    # quarter of the largest expert's
    scale = np.abs(ref["dW_e"]).max()
    for e in range(E):
        err = np.abs(dWe[e].double().numpy() - ref["dW_e"][e]).max()
        assert err <= 2e-2 * max(np.abs(ref["dW_e"][e]).max(), scale / 4), (e, err)
        if not np.any(idx.numpy() == e):
            assert float(dWe[e].abs().max()) == 0.0
    assert np.abs(dWr.double().numpy() - ref["dW_r"]).max() <= 2e-2 * np.abs(ref["dW_r"]).max()
