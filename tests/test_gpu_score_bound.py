"""The scorer's in-flight bound, candidate lists and evened-out tiles.

Each CTA publishes its j-th best first-tile score and lists only what reaches
the r-th largest of them: sizes where j is 1, 2 .. 8, 9 .. 32 and where no bound
is taken; stores sorted by score, which fill every list and turn it into a heap;
exact ties; tiles of 64 .. 256 rows; scans long enough for the bound to be taken
again from the lists (before tiles 2, 6, 20 of a CTA's more than 8, 24, 80), for
each range of j on each kernel.
"""
import pytest
import torch

import paper_2606_11660_gb300 as bg
from paper_2606_11660_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _search(store, queries, k, least=False):
    N, K = store.shape
    Q = queries.shape[0]
    ws = bg.workspace_tensor(bg.bergson_score_topk_workspace(N, K, Q, k), DEV)
    ws.fill_(0xA5)                                    # contents on entry are ignored
    s = torch.full((Q, k), float("nan"), device=DEV)
    i = torch.full((Q, k), -7, dtype=torch.int64, device=DEV)
    fn = bg.bergson_score_bottomk if least else bg.bergson_score_topk
    fn(store, N, K, queries, k, s, i, ws)
    assert bg.bergson_sync_status() == bg.BERGSON_OK, bg.bergson_last_error()
    return s, i


def _queries(Q, seed):
    # entries +-1: the norm is 8 and the unit query exact in fp16, so that the
    # reference needs no allowance for how a query entry was rounded
    return torch.sign(wl.gaussian_rows(Q, 64, seed, DEV))


def _check(store, queries, k, s, i, least=False):
    q = queries.double()
    q = q / q.norm(dim=1, keepdim=True)
    for a in range(0, q.shape[0], 64):
        S = q[a:a + 64] @ store.double().T
        want = S.topk(k, dim=1, largest=not least).values
        got = s[a:a + 64].double()
        assert (got - want).abs().max() <= 2e-6       # sums of K fp16 products in fp32
        assert (S.gather(1, i[a:a + 64]) - got).abs().max() <= 2e-6
    assert all(len(set(r.tolist())) == k for r in i[:8].cpu())


def _rows(N, K, seed):
    return torch.nn.functional.normalize(wl.gaussian_rows(N, K, seed, DEV), dim=1).half()


@pytest.mark.parametrize("N,Q,topk", [
    (9_000, 5, 1), (40_000, 3, 10), (40_000, 100, 152), (40_000, 7, 300), (40_000, 128, 1000),
    (39_000, 129, 100), (39_000, 200, 500), (39_000, 300, 40), (39_000, 300, 300),
    (39_000, 1024, 1000), (20_011, 16, 1024), (300, 3, 20), (64 * 152 + 1, 2, 9), (500, 1, 400),
    (12_000, 3000, 300),
])
def test_bound_classes(N, Q, topk):
    store, queries = _rows(N, 64, N + Q), _queries(Q, topk)
    least = topk % 2 == 1
    s, i = _search(store, queries, topk, least)
    _check(store, queries, topk, s, i, least)


@pytest.mark.parametrize("Q,topk", [(3, 5), (3, 200), (140, 30), (300, 60)])
@pytest.mark.parametrize("ascending", [True, False])
def test_sorted_store_fills_every_list(Q, topk, ascending):
    N = 152 * 256 * 3 // (1 if Q < 129 else 2 if Q <= 256 else 4) + 77
    queries = _queries(1, 5).repeat(Q, 1)             # one order suits them all: an entry flipped
    queries[torch.arange(1, Q), torch.arange(1, Q) % 64] *= -1
    store = _rows(N, 64, 6)
    order = (store.double() @ queries[0].double()).argsort(descending=not ascending)
    store = store[order].contiguous()
    s, i = _search(store, queries, topk)
    _check(store, queries, topk, s, i)


@pytest.mark.parametrize("Q,topk", [(2, 150), (150, 40), (300, 40)])
def test_equal_rows_come_in_index_order(Q, topk):
    store = _rows(1, 64, 8).expand(30_000, 64).contiguous()
    s, i = _search(store, _queries(Q, 9), topk)
    assert torch.equal(i, torch.arange(topk, device=DEV).expand(Q, topk))
    assert (s == s[:, :1]).all()


@pytest.mark.parametrize("Q,topk,tiles,j", [
    (2, 100, 10, (1, 1)), (1, 30, 82, (1, 1)), (2, 300, 26, (2, 8)), (3, 1024, 10, (9, 32)),
    (140, 60, 26, (1, 1)), (200, 200, 10, (2, 8)), (200, 800, 26, (9, 32)),     # pairs, one tile
    (300, 40, 26, (1, 1)), (300, 100, 26, (2, 8)), (1024, 1000, 10, (9, 32)),   # pairs, two tiles
])
def test_bound_taken_again(Q, topk, tiles, j):
    groups = 1 if Q < 129 else 2 * -(-Q // (256 if Q <= 256 else 512))
    N = 256 * tiles * (152 // groups)
    launch = bg.bergson_debug_score_launches(N, 64, Q, topk, 152)
    assert len(launch) == 1 and launch[0]["n_qg"] == groups
    assert j[0] <= launch[0]["bound_j"] <= j[1]
    assert -(-launch[0]["n_tiles"] // launch[0]["cpg"]) == tiles > 8
    store, queries = _rows(N, 64, tiles), _queries(Q, 3)
    store[N // 2] = float("nan")                      # a row that is never found
    s, i = _search(store, queries, topk)
    assert not (i == N // 2).any()
    store[N // 2] = 0
    _check(store, queries, topk, s, i)
