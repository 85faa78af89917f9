"""The planner's line for cutting per-token score slots, through the workspace it asks for (CPU)."""
import pytest
import torch

import paper_2606_11660_gb300 as bg


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
