"""Workspace queries over ranges of sizes, without a device: they read nothing of a handle but its
configuration and the SM count, which lead it."""
import ctypes
import random

import pytest

from paper_2603_06938_b200 import binding as sb
from paper_2603_06938_b200 import build as sbuild

SMS = 148


def handle(F, H, G, E, k, chunk, P=64, N=128, dtype=sb.DTYPE_BF16):
    sbuild.build()
    block = (ctypes.c_int32 * 4096)(F, H, P, N, G, E, k, chunk, dtype, 0, 0, SMS)
    return block, ctypes.cast(block, ctypes.c_void_p)


LAYERS = [(768, 24, 1, 8, 2, 256), (2048, 64, 1, 8, 2, 128), (1152, 36, 2, 16, 4, 256), (64, 3, 1, 4, 1, 64),
          (768, 96, 1, 64, 3, 128), (512, 2, 2, 1, 1, 256), (2048, 160, 1, 8, 2, 128)]


@pytest.mark.parametrize("name", ["workspace", "ssd_slots_workspace", "block_workspace", "backward_workspace",
                                  "shard_workspace", "host_workspace"])
@pytest.mark.parametrize("layer", LAYERS)
def test_smaller_calls_need_no_more(name, layer):
    """128-token tiles decide the segments: every tile count of a sequence, then batches."""
    keep, h = handle(*layer)
    need = getattr(sb.lib(), f"swimba_{name}_bytes")
    lengths = [1, 100] + list(range(128, 128 * 200, 128)) + list(range(25600, 140000, 3712))
    for B in (1, 2, 3, 7):
        sizes = [need(h, B, L) for L in lengths]
        assert sizes == sorted(sizes)
    for L in (90, 300, 1500, 2432, 5376, 24704, 100000):
        sizes = [need(h, B, L) for B in range(1, 80)]
        assert sizes == sorted(sizes)


def test_segment_states_fit_what_is_reserved():
    """The forward's regions, by the sizes that include/swimba.h names, with the states of the segments that
    the call really makes."""
    up = lambda v: (v + 255) // 256 * 256
    rnd = random.Random(5)
    need, segments = sb.lib().swimba_workspace_bytes, sb.lib().swimba_ssd_segments
    for F, H, G, E, k, chunk in LAYERS:
        keep, h = handle(F, H, G, E, k, chunk)
        S, PN = 2 * G * 128, 64 * 128
        for _ in range(1500):
            B, L = rnd.randint(1, 20), int(2 ** rnd.uniform(0, 17))
            T, tiles, nseg = B * L, (L + 127) // 128, segments(h, B, L)
            size = up(T * S * 2) + 2 * up(T * k * 4) + up(256 + up(E * T * 4) + (up(T * k * S * 2) if k > 2 else 0))
            size += up(B * H * tiles * 512) + up(B * H * tiles * 1040)
            if nseg > 1:
                size += B * nseg * H * (PN + 1) * 4
            assert size <= need(h, B, L), (B, L, nseg)


@pytest.mark.parametrize("F,H,E,k,chunk,B,L", [(768, 64, 4, 1, 256, 4, 9956), (768, 32, 16, 2, 256, 5, 9924),
                                               (768, 48, 8, 2, 128, 9, 600), (2048, 64, 8, 2, 128, 4, 9984)])
def test_host_workspace_serves_every_slice(F, H, E, k, chunk, B, L):
    """Behind the staged tensors (u, x, dt, y, two state buffers, routing) the forward's workspace for any slice:
    up to an eighth of the sequences, or a run of tokens of one."""
    up = lambda v: (v + 255) // 256 * 256
    keep, h = handle(F, H, 1, E, k, chunk)
    T, HP = B * L, H * 64
    staged = up(T * F * 2) + 2 * up(T * HP * 2) + up(T * H * 4) + 2 * up(B * HP * 128 * 4) + 2 * up(T * k * 4)
    left = sb.lib().swimba_host_workspace_bytes(h, B, L) - staged
    assert max(sb.lib().swimba_workspace_bytes(h, n, L) for n in range(1, (B + 7) // 8 + 1)) <= left
    assert max(sb.lib().swimba_workspace_bytes(h, 1, n) for n in range(1, L + 1)) <= left


@pytest.mark.parametrize("F,G,E,k,dtype", [(2048, 1, 8, 2, "bf16"), (768, 1, 16, 4, "bf16"), (4096, 2, 16, 8, "bf16"),
                                           (96, 1, 4, 1, "bf16"), (2048, 1, 64, 3, "bf16"), (256, 1, 8, 3, "fp32")])
def test_smaller_decode_batches_need_no_more(F, G, E, k, dtype):
    keep, h = handle(F, 8, G, E, k, 128, dtype=sb.DTYPE_FP32 if dtype == "fp32" else sb.DTYPE_BF16)
    sizes = [sb.lib().swimba_decode_workspace_bytes(h, B) for B in range(1, 1200)]
    assert sizes == sorted(sizes)
    if E <= 16 and dtype == "bf16":      # the small front end: k fp32 rows per sequence up to B = 4
        assert sizes[3] >= 4 * k * 256 * G * 4
    # larger batches take no slots of fp32 rows: one row of streams, the lists, 16-bit slots where k > 2
    S = 256 * G
    assert sizes[1100] - sizes[256] <= (1100 - 256) * (4 * S + (2 * k * S if k > 2 else 0) + 4 * E + 8 * k) + 4096
