"""The products on CTA pairs at the edges of their tiles: rows of an expert around 128 and 256, column
tiles that end inside 256 columns, feature counts that are no multiple of 64, every expert count, and the
three ways a row leaves (added, stored per slot and mixed, stored)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_06938_b200 import binding as sb
from paper_2603_06938_b200 import synth

import helpers as hp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,F,G,N,E,k", [(2048, 64, 1, 128, 8, 1), (1023, 72, 1, 144, 3, 2), (1030, 136, 2, 128, 5, 3),
                                         (2305, 192, 1, 16, 64, 2), (4101, 328, 1, 80, 16, 2), (2049, 64, 1, 256, 1, 1)])
def test_projection_and_mix_match_oracle(T, F, G, N, E, k):
    cfg = synth.LayerConfig("pair", "bf16", 1, T, F, 2 * G, 8, N, G, E, k, 64)
    inp = synth.make_inputs(cfg, seed=500 + T)
    h = hp.create_handle(cfg, None, sb.FLAG_CHECK_INDICES)
    w, keep = hp.device_weights(inp)
    BC, raw = hp.with_canary((T, cfg.S), torch.bfloat16, float("nan"))
    idx = torch.full((T, k), -1, dtype=torch.int32, device="cuda")
    wt = torch.full((T, k), float("nan"), device="cuda")
    ws = torch.empty(sb.swimba_workspace_bytes(h, 1, T), dtype=torch.uint8, device="cuda")
    sb.swimba_route_mix(h, w, hp.dev(inp["u"][0]), T, BC, idx, wt, ws)
    assert sb.swimba_status(h) == 0, sb.swimba_last_error(h)
    assert hp.canary_intact(raw)
    sb.swimba_destroy(h)
    u, W_e = synth.f64(inp["u"][0]), synth.f64(inp["W_e"])
    ii, ww = idx.cpu().numpy(), wt.cpu().double().numpy()
    slots = ww[..., None] * np.take_along_axis(oracle.expert_streams(u, W_e), ii[..., None].astype(np.int64), 1)
    # bf16 keeps eight significant bits: storing a value costs up to 2^-8 of it.  One slot is stored once;
    # of several, each is stored and their sum is (first order 2^-8 (sum |s_j| + |sum s_j|), second-order
    # terms within the extra 1 %).  fp32 accumulation adds at most F 2^-24 of the sum of the absolute
    # products, which is at most sqrt(F) times a typical entry here.
    bound = 1.01 * 2.0 ** -8 * (np.abs(slots.sum(1)) + (np.abs(slots).sum(1) if k > 1 else 0.0)) \
        + F ** 1.5 * 2.0 ** -24 * np.abs(slots).max()
    err = np.abs(BC.cpu().double().numpy() - slots.sum(1))
    assert np.all(err <= bound), float((err - bound).max())
