"""The workspace of a projection call: one sized for a batch serves smaller ones (CPU)."""
import ctypes
import random

import pytest

import paper_2606_11660_gb300 as bg
from paper_2606_11660_gb300 import workloads as wl

FAKE = 0x7F0000000000                                 # aligned, never dereferenced
DIMS = {"tiny": [(64, 64)]}
for _name in ("pythia160m", "pythia1b4", "llama8b"):
    DIMS[_name] = [(s.d_in, s.d_out) for s in wl.COLLECT_WORKLOADS[_name].block_modules(0)]


def _layers(dims, k):
    arr = (bg.bergson_layer * len(dims))()
    for i, (d_in, d_out) in enumerate(dims):
        arr[i] = bg.bergson_layer(A=FAKE + (i << 28), G=FAKE + (i << 28), d_in=d_in, d_out=d_out,
                                  k_in=k[0], k_out=k[1], out_col_offset=i * k[0] * k[1])
    return arr


def _query(arr, n, B, T):
    ws = ctypes.c_size_t()
    assert bg.lib().bergson_project_grads_workspace(arr, n, B, T, ctypes.byref(ws)) == bg.BERGSON_OK
    return ws.value


def _status(arr, n, B, T, ws_bytes, k):
    """What the call answers: EDEVICE_TIMEOUT, injected behind the workspace check, or EWORKSPACE."""
    ld = len(arr) * k[0] * k[1]
    bg.lib().bergson_debug_inject_status(bg.BERGSON_EDEVICE_TIMEOUT, 1)
    try:
        return bg.lib().bergson_project_grads(arr, n, B, T, None, FAKE, ld, FAKE, ws_bytes, None)
    finally:
        bg.lib().bergson_debug_inject_status(0, 0)


# (family, blocks, k, batch the workspace is sized for, smaller batch, its modules)
BATCHES = [
    ("pythia160m", 1, (16, 64), (39, 121), (27, 65), 4),
    ("pythia160m", 3, (16, 16), (19, 12), (8, 4), 12),
    ("tiny", 3, (16, 32), (44, 20), (37, 4), 1),
    ("tiny", 6, (16, 16), (8, 360), (7, 197), 6),
    ("tiny", 3, (16, 16), (2, 2075), (1, 1623), 3),
    ("tiny", 1, (32, 16), (17, 1330), (12, 418), 1),
    ("pythia160m", 2, (32, 16), (9, 170), (7, 10), 8),
    ("pythia1b4", 1, (64, 32), (11, 628), (6, 202), 4),
    ("pythia160m", 6, (32, 64), (8, 92), (5, 59), 24),
    ("pythia1b4", 3, (32, 16), (2, 721), (2, 345), 12),
]


@pytest.mark.parametrize("family,blocks,k,big,small,n", BATCHES)
def test_workspace_of_a_batch_serves_a_smaller_one(family, blocks, k, big, small, n):
    arr = _layers(DIMS[family] * blocks, k)
    size = _query(arr, len(arr), *big)
    assert _status(arr, n, *small, size, k) == bg.BERGSON_EDEVICE_TIMEOUT


def test_queried_size_is_taken_and_projections_alone_are_not():
    r = random.Random(2)
    for _ in range(200):
        k = (r.choice([16, 32, 64]), r.choice([16, 32, 64]))
        arr = _layers(DIMS[r.choice(list(DIMS))] * r.choice([1, 2, 7]), k)
        B, T = int(2 ** r.uniform(0, 5)), int(2 ** r.uniform(3, 12))
        size = _query(arr, len(arr), B, T)
        assert _status(arr, len(arr), B, T, size, k) == bg.BERGSON_EDEVICE_TIMEOUT
        p = sum(4 * (k[0] * l.d_in + k[1] * l.d_out) for l in arr)     # P'
        assert _status(arr, len(arr), B, T, p, k) == bg.BERGSON_EWORKSPACE


@pytest.mark.parametrize("family,blocks,k,B,T", [("llama8b", 7, (16, 16), 1, 129),
                                                 ("llama8b", 7, (16, 16), 4, 129),
                                                 ("pythia1b4", 12, (32, 32), 2, 512)])
def test_large_projections_leave_the_slots_of_a_small_launch(family, blocks, k, B, T):
    # more than the allocation-free call's 32 MB, for P' mostly: slots of one tile all the same
    arr = _layers(DIMS[family] * blocks, k)
    assert _query(arr, len(arr), B, T) > 32 << 20
    n = [ctypes.c_int64() for _ in range(4)]
    assert bg.lib().bergson_debug_project_plan(arr, len(arr), B, T, *map(ctypes.byref, n)) == 0
    assert n[0].value == len(arr) * B * -(-T // 128)


@pytest.mark.parametrize("family,blocks,k,B,T", [("llama8b", 5, (16, 16), 2, 512),
                                                 ("llama8b", 2, (32, 32), 8, 300),
                                                 ("pythia1b4", 6, (64, 16), 1, 129)])
def test_allocation_free_call_takes_what_its_scratch_can_do(family, blocks, k, B, T):
    arr = _layers(DIMS[family] * blocks, k)
    assert _query(arr, len(arr), B, T) > 32 << 20     # with the finest cut
    st = bg.lib().bergson_project_grads_noalloc(arr, len(arr), B, T, None, FAKE,
                                                len(arr) * k[0] * k[1], None)
    assert st == bg.BERGSON_EINVAL                    # FAKE is no device memory; not EWORKSPACE
    assert "not device memory" in bg.bergson_last_error()
