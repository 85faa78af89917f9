"""Per-token scores of few, wide slots: slots cut into pieces, query blocks behind the piece sums."""
import numpy as np
import pytest
import torch

import paper_2606_11660_gb300 as bg
from oracle import bergson_oracle as orc
from paper_2606_11660_gb300 import workloads as wl
from tests._util import make_layers, np32

pytestmark = pytest.mark.gpu
DEV = "cuda"
B, T = 2, 150


def _coarse_bytes(specs, k, n_queries):
    """P' (hi and lo bf16) and the partials, each region within 256 bytes, and 64 KB of records."""
    n = 0
    for s in specs:
        n += 4 * (k[0] * s.d_in + k[1] * s.d_out) + 4 * n_queries * B * T
    return n + 65536


@pytest.mark.parametrize("n_queries", [1, 40])
@pytest.mark.parametrize("k", [(16, 16), (32, 16), (16, 32), (32, 32), (16, 64), (64, 16), (32, 64)])
def test_pieces(k, n_queries):
    specs = [wl.ModuleSpec("wide", 3208, 3272), wl.ModuleSpec("small", 64, 200)]
    gl, ol, ld = make_layers(specs, B, T, [k] * 2, base_seed=5, data_seed=n_queries, rc=True)
    g = wl.generator(11, "cpu")
    mask = (torch.rand((B, T), generator=g) > 0.3).to(torch.uint8)
    mask[0, 32:64] = 0                     # a slice that is not read
    mask[1, 128:] = 0                      # and a tile
    queries = torch.randn((n_queries, ld + (n_queries & 1)), generator=g)   # odd row strides too
    total = bg.bergson_token_scores_workspace(gl, B, T, n_queries)
    coarse = _coarse_bytes(specs, k, n_queries)
    assert total > coarse + 4 * 2 * B * 128 * (k[0] + k[1])    # every piece's projections
    want = orc.token_scores(ol, mask.numpy(), queries.numpy())
    scale = np.abs(want).max(axis=(1, 2), keepdims=True)
    for size in (total, coarse):           # a workspace without room for pieces still serves
        ws = bg.workspace_tensor(size, DEV)
        out = torch.full((n_queries, B, T), float("nan"), device=DEV)
        bg.bergson_token_scores(gl, B, T, mask.to(DEV), queries.to(DEV), out, ws)
        assert bg.bergson_sync_status() == bg.BERGSON_OK, bg.bergson_last_error()
        got = np32(out).astype(np.float64)
        assert np.all(got[:, mask.numpy() == 0] == 0.0)
        # bf16 hi + lo projections: 1e-4 of a query's largest score, as for whole slots
        assert np.all(np.abs(got - want) <= 1e-4 * scale + 1e-12)
