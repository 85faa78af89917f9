"""Calls whose workspace has only the least size: coarsely cut collections, searches without a bound."""
import numpy as np
import pytest
import torch

import paper_2606_11660_gb300 as bg
from oracle import bergson_oracle as orc
from paper_2606_11660_gb300 import workloads as wl
from tests._util import make_layers, np32, rel_frobenius

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _least_workspace(call, most):
    """The least size `call` takes, by its status injected behind the workspace check."""
    lo, hi = 0, most
    while lo < hi:
        mid = (lo + hi) // 2 // 256 * 256
        bg.lib().bergson_debug_inject_status(bg.BERGSON_EDEVICE_TIMEOUT, 1)
        try:
            call(bg.workspace_tensor(mid, DEV)[:mid])
            raise AssertionError("no status")
        except bg.BergsonError as e:
            assert e.status in (bg.BERGSON_EDEVICE_TIMEOUT, bg.BERGSON_EWORKSPACE)
            ok = e.status == bg.BERGSON_EDEVICE_TIMEOUT
        finally:
            bg.lib().bergson_debug_inject_status(0, 0)
        lo, hi = (lo, mid) if ok else (mid + 256, hi)
    return hi


@pytest.mark.parametrize("dims,B,T,k", [
    ([(3208, 3272), (64, 200)], 2, 150, (16, 16)),     # pieces of one-tile slots, or of whole ones
    ([(768, 2304), (768, 768)], 3, 333, (32, 16)),
    ([(768, 768)] * 3, 4, 500, (16, 16)),
    ([(4096, 1024)], 1, 700, (32, 32)),
])
def test_collection_with_room_for_the_coarse_cut_only(dims, B, T, k):
    specs = [wl.ModuleSpec(f"m{i}", d_in, d_out) for i, (d_in, d_out) in enumerate(dims)]
    gl, ol, ld = make_layers(specs, B, T, [k] * len(specs), base_seed=7, data_seed=B, rc=True)
    mask = (torch.rand((B, T), generator=wl.generator(T, "cpu")) > 0.3).to(torch.uint8)
    out = torch.full((B, ld), float("nan"), device=DEV)
    md = mask.to(DEV)
    size = bg.bergson_project_grads_workspace(gl, B, T)
    least = _least_workspace(lambda ws: bg.bergson_project_grads(gl, B, T, md, out, ws), size)
    assert least < size
    want = orc.project_grads(ol, mask.numpy(), ld)
    for n in (size, least):
        out.fill_(float("nan"))
        bg.bergson_project_grads(gl, B, T, md, out, bg.workspace_tensor(n, DEV)[:n])
        assert bg.bergson_sync_status() == bg.BERGSON_OK, bg.bergson_last_error()
        # P' in bf16 hi + lo: 2^-16 an entry
        assert rel_frobenius(np32(out).astype(np.float64), want).max() < 2.0 ** -14


@pytest.mark.parametrize("N,Q,topk", [(20_011, 3, 3), (40_000, 128, 4), (39_000, 140, 4),
                                      (300, 2, 1), (39_000, 300, 2), (200_000, 600, 1)])
@pytest.mark.parametrize("least", [False, True])
def test_search_without_room_for_the_published_scores(N, Q, topk, least):
    # they lie behind the lists for topk < 5: the former size has no room, and takes no bound
    store = torch.nn.functional.normalize(wl.gaussian_rows(N, 64, N, DEV), dim=1).half()
    queries = torch.sign(wl.gaussian_rows(Q, 64, Q, DEV))
    size = bg.bergson_score_topk_workspace(N, 64, Q, topk)
    fn = bg.bergson_score_bottomk if least else bg.bergson_score_topk
    res = []
    for n in (size, size - 152 * 128 * (1 if Q <= 256 else 2) * 2):
        ws = bg.workspace_tensor(n, DEV)[:n]
        ws.fill_(0x5A)
        s = torch.full((Q, topk), float("nan"), device=DEV)
        i = torch.full((Q, topk), -7, dtype=torch.int64, device=DEV)
        fn(store, N, 64, queries, topk, s, i, ws)
        assert bg.bergson_sync_status() == bg.BERGSON_OK, bg.bergson_last_error()
        res.append((s, i))
    assert torch.equal(res[0][0], res[1][0]) and torch.equal(res[0][1], res[1][1])
    q = queries.double() / 8.0
    for a in range(0, Q, 64):
        want = (q[a:a + 64] @ store.double().T).topk(topk, dim=1, largest=not least).values
        assert (res[1][0][a:a + 64].double() - want).abs().max() <= 2e-6
    with pytest.raises(bg.BergsonError) as e:
        fn(store, N, 64, queries, topk, *res[0], ws[:n - 256])
    assert e.value.status == bg.BERGSON_EWORKSPACE
