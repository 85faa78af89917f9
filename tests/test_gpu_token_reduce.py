"""The sum of per-token partials over modules: four tokens a thread or one, batches of eight modules."""
import numpy as np
import pytest
import torch

import paper_2606_11660_gb300 as bg
from oracle import bergson_oracle as orc
from paper_2606_11660_gb300 import workloads as wl
from tests._util import make_layers, np32

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("n_mods", [1, 8, 9, 17])
@pytest.mark.parametrize("B,T,shift", [(1, 1, 0), (3, 7, 0), (3, 7, 1), (2, 130, 0), (4, 33, 1)])
def test_module_sums(n_mods, B, T, shift):
    specs = [wl.ModuleSpec(f"m{i}", 16, 24) for i in range(n_mods)]
    gl, ol, ld = make_layers(specs, B, T, [(16, 16)] * n_mods, base_seed=3, data_seed=n_mods, rc=True)
    g = wl.generator(9, "cpu")
    queries = torch.randn((3, ld), generator=g)
    mask = (torch.rand((B, T), generator=g) > 0.3).to(torch.uint8)
    ws = bg.workspace_tensor(bg.bergson_token_scores_workspace(gl, B, T, 3), DEV)
    # shift: results that start off a 16-byte boundary
    out = torch.full((3 * B * T + shift,), float("nan"), device=DEV)[shift:].view(3, B, T)
    bg.bergson_token_scores(gl, B, T, mask.to(DEV), queries.to(DEV), out, ws)
    assert bg.bergson_sync_status() == bg.BERGSON_OK, bg.bergson_last_error()
    got = np32(out).astype(np.float64)
    assert np.all(got[:, mask.numpy() == 0] == 0.0)
    # A module's sum against the 64-bit sum: n_mods - 1 roundings of partial sums, each at most
    # 2^-24 of the sum of magnitudes, far below the partials' own error (bf16-split projections,
    # 1e-4 of the largest score as in the other per-token tests).
    want = orc.token_scores(ol, mask.numpy(), queries.numpy())
    scale = np.abs(want).max(axis=(1, 2), keepdims=True)
    assert np.all(np.abs(got - want) <= 1e-4 * scale + 1e-12)
