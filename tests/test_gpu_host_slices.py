"""The host-buffer forward with a last slice shorter than the others, in tokens and in sequences, on exactly
the workspace it asks for, against the device entry point."""
import pytest
import torch

from paper_2603_06938_b200 import binding as sb
from paper_2603_06938_b200 import synth

import helpers as hp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,H,k,chunk", [(6, 3212, 32, 1, 64), (9, 528, 8, 2, 256)])
def test_uneven_slices_match_device_entry_point(B, L, H, k, chunk):
    cfg = synth.LayerConfig("slices", "bf16", B, L, 64, H, 64, 128, 1, 4, k, chunk)
    inp = synth.make_inputs(cfg, seed=70 + B)
    want = hp.gpu_forward(cfg, inp)
    h = hp.create_handle(cfg)
    w, keep = hp.device_weights(inp)
    ws, ws_raw = hp.with_canary((sb.swimba_host_workspace_bytes(h, B, L),), torch.uint8, 0)
    u, x, dt = inp["u"].pin_memory(), inp["x"].pin_memory(), inp["dt"].pin_memory()
    y, hf = torch.empty_like(x).pin_memory(), torch.empty(B, H, 64, 128).pin_memory()
    idx = torch.empty(B, L, k, dtype=torch.int32).pin_memory()
    sb.swimba_forward_host(h, w, u, x, dt, B, L, y, hf, idx, None, ws)
    assert sb.swimba_status(h) == 0
    # (slices are cut into other segments than the whole call: equal within the parity tolerance)
    tol_y, tol_h = hp.tolerances(cfg)
    assert hp.max_rel(y.double().numpy(), want["y"].double().numpy()) <= tol_y
    assert hp.max_rel(hf.numpy(), want["h_final"].numpy()) <= tol_h
    assert torch.equal(idx, want["idx"])
    assert hp.canary_intact(ws_raw)
    sb.swimba_destroy(h)
