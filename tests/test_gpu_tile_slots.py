"""Collections in slots of one tile: stages of one tile, whole slots and pieces, masks and biases."""
import numpy as np
import pytest
import torch

import paper_2606_11660_gb300 as bg
from oracle import bergson_oracle as orc
from paper_2606_11660_gb300 import workloads as wl
from tests._util import make_layers, np32, rel_frobenius, run_project

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("T", [1, 31, 128, 129, 300])
@pytest.mark.parametrize("k", [(16, 16), (16, 32), (32, 16), (32, 32)])
def test_one_tile_slots(k, T):
    B = 3
    specs = [wl.ModuleSpec("whole", 200, 136), wl.ModuleSpec("cut", 1096, 904)]
    gl, ol, ld = make_layers(specs, B, T, [k] * 2, base_seed=2, data_seed=T, rc=True)
    n_tiles = (T + 127) // 128
    slots, items, pieces, _ = bg.bergson_debug_project_plan(gl, B, T)
    assert slots == 2 * B * n_tiles and 0 < pieces
    g = wl.generator(13, "cpu")
    mask = (torch.rand((B, T), generator=g) > 0.2).to(torch.uint8)
    mask[:, 0] = 1
    mask[1, 96:256] = 0                    # slices, and (T = 300) a tile that is not read
    for m in (None, mask):
        got = np32(run_project(gl, B, T, None if m is None else m.to(DEV), ld)).astype(np.float64)
        want = orc.project_grads(ol, None if m is None else m.numpy(), ld)
        # bf16 hi + lo projections, 2^-16 an entry a side: 1e-4, as in the other parity tests
        assert rel_frobenius(got, want).max() <= 1e-4
