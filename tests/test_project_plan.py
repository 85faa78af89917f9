"""The lines of the projection planner: slots, and when they are cut into pieces (CPU)."""
import pytest
import torch

import paper_2606_11660_gb300 as bg
from paper_2606_11660_gb300 import workloads as wl
from tests.test_abi import _block_layers, _plan


def _layers(dims, B, T, k):
    out, off = [], 0
    for i, (d_in, d_out) in enumerate(dims):
        out.append(bg.Layer(torch.zeros(B, T, d_in, dtype=torch.bfloat16),
                            torch.zeros(B, T, d_out, dtype=torch.bfloat16), k[0], k[1], 2 * i,
                            2 * i + 1, None, None, off, bg.BERGSON_PROJ_GAUSSIAN))
        off += k[0] * k[1]
    return out


def _extra(dims, B, T, k, q):
    """Workspace beyond P' and the partials."""
    n = sum(4 * (k[0] * i + k[1] * o) + 4 * q * B * T for i, o in dims)
    return bg.bergson_token_scores_workspace(_layers(dims, B, T, k), B, T, q) - n


@pytest.mark.parametrize("dims,B,T,k,q,cut", [
    ([(6016, 4096)], 1, 100, (16, 16), 1, True),       # 158 units, a share of 1: 64 + 0.75 q
    ([(6016, 4096)], 1, 100, (16, 16), 120, True),     # 157 > 154
    ([(6016, 4096)], 1, 100, (16, 16), 128, False),    # 157 < 160
    ([(2048, 2048)], 1, 100, (16, 16), 1, False),      # 64 units: 63.6 < 64.75
    ([(2112, 2112)], 1, 100, (16, 16), 1, True),       # 66 units: 65.6 > 64.75
    ([(6016, 4096)], 1, 100, (32, 64), 1, True),       # one query a block
    ([(6016, 4096)], 1, 100, (64, 32), 1, False),      # CUDA cores: whole slots
    ([(6016, 4096)], 1, 100, (64, 64), 1, False),
])
def test_cut(dims, B, T, k, q, cut):
    tile_rows = 4 * B * 128 * (k[0] + k[1])            # one piece a side, one tile
    extra = _extra(dims, B, T, k, q)
    assert (extra >= tile_rows) == cut


@pytest.mark.parametrize("name,blocks,B,T,k,tiles,cut", [
    ("pythia160m", 2, 7, 333, 16, 1, False),     # one-tile slots; 60 units to a share of 53
    ("pythia160m", 1, 1, 300, 16, 1, True),      # 60 to 4
    ("llama8b", 1, 2, 1024, 16, 1, True),
    ("llama8b", 1, 8, 4096, 16, 4, True),        # a large share: pieces as before
    ("pythia160m", 12, 16, 129, 16, 1, False),   # two tiles would half fill a stage
    ("pythia160m", 9, 29, 257, 16, 4, False),    # three of four: one slot an example
    ("pythia1b4", 1, 16, 2048, 32, 2, False),
])
def test_slots_of_collections(name, blocks, B, T, k, tiles, cut):
    cfg = wl.COLLECT_WORKLOADS[name]
    specs = [s for b in range(blocks) for s in cfg.block_modules(b)]
    slots, items, pieces, _ = _plan(_block_layers(specs, k), B, T)
    n_tiles = (T + 127) // 128
    assert slots == len(specs) * B * max(1, -(-n_tiles // tiles))
    assert (pieces > 0) == cut
