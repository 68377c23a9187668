"""States updated in place (h_final is h0) against the same call with two buffers, where several blocks of one
launch read the given and write the final state of a sequence: segments, leading tiles, clusters."""
import pytest
import torch

from paper_2603_06938_b200 import binding as sb
from paper_2603_06938_b200 import synth

import helpers as hp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,B,L,H,P,N", [("bf16", 1, 2177, 6, 64, 128), ("bf16", 4, 1500, 8, 64, 128),     # segments
                                             ("bf16", 25, 641, 6, 64, 128),                                    # leading tiles
                                             ("fp32", 3, 300, 4, 32, 16)])                                     # cluster
def test_in_place_forward(dtype, B, L, H, P, N):
    cfg = synth.LayerConfig("inplace", dtype, B, L, 64, H, P, N, 1, 4, 2, 128, h0_std=0.2)
    inp = synth.make_inputs(cfg, seed=50 + B)
    want = hp.gpu_forward(cfg, inp)
    h = hp.create_handle(cfg)
    w, keep = hp.device_weights(inp)
    state, y = hp.dev(inp["h0"]), torch.empty_like(hp.dev(inp["x"]))
    ws = torch.empty(sb.swimba_workspace_bytes(h, B, L), dtype=torch.uint8, device="cuda")
    sb.swimba_forward(h, w, hp.dev(inp["u"]), hp.dev(inp["x"]), hp.dev(inp["dt"]), state, B, L, y, state, None, None, ws)
    assert sb.swimba_status(h) == 0
    if B == 25:         # leading tiles are evaluated by other blocks when there are two buffers: rounding differs
        tol_y, tol_h = hp.tolerances(cfg)
        assert hp.max_rel(y.cpu().double().numpy(), want["y"].double().numpy()) <= tol_y
        assert hp.max_rel(state.cpu().numpy(), want["h_final"].numpy()) <= tol_h
    else:
        assert torch.equal(y.cpu(), want["y"]) and torch.equal(state.cpu(), want["h_final"])
    sb.swimba_destroy(h)


@pytest.mark.parametrize("lens", [[1300, 1, 0, 700, 3, 40, 5], [4, 129, 1], [0, 0]])
def test_in_place_packed(lens):
    cfg = synth.LayerConfig("inplace", "bf16", 1, max(sum(lens), 1), 64, 4, 64, 128, 1, 4, 2, 128)
    inp = synth.make_inputs(cfg, seed=60)
    gen = torch.Generator().manual_seed(61)
    h0 = 0.2 * torch.randn(len(lens), cfg.H, cfg.P, cfg.N, generator=gen)
    cu = [sum(lens[:i]) for i in range(len(lens) + 1)]
    h = hp.create_handle(cfg)
    w, keep = hp.device_weights(inp)
    u, x, dt = (hp.dev(inp[n][0]) for n in ("u", "x", "dt"))
    ws = torch.empty(max(sb.swimba_packed_workspace_bytes(h, cu), 16), dtype=torch.uint8, device="cuda")
    got = []
    for in_place in (False, True):
        state = h0.cuda()
        hf = state if in_place else torch.empty_like(state)
        y = torch.zeros_like(x)
        sb.swimba_forward_packed(h, w, u, x, dt, state, cu, y, hf, None, None, ws)
        assert sb.swimba_status(h) == 0
        got.append((y.cpu(), hf.cpu()))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    sb.swimba_destroy(h)
