"""The score launches as they are made: tiles, grid and bound (CPU)."""
import random

import pytest

import paper_2606_11660_gb300 as bg

K = 64
SIZES = [(20_011, 3, 10, 152), (250_007, 100, 100, 152), (4_000_000, 1024, 100, 152),
         (300_000, 1024, 300, 152), (39_000, 129, 100, 152), (39_000, 300, 40, 152),
         (500, 1, 400, 152), (1, 1, 1, 152), (64 * 152 + 1, 2, 9, 152), (12_000, 3000, 300, 152),
         (10_000, 16, 64, 3), (1_000_000, 41_000, 100, 160), (30_000, 260, 1024, 148)]


def _random_sizes():
    r = random.Random(11)
    for _ in range(300):
        N = int(10 ** r.uniform(0, 6.6))
        yield N, int(10 ** r.uniform(0, 4.6)), min(N, int(10 ** r.uniform(0, 3.01))), r.choice(
            [2, 37, 148, 152, 153, 160, 200])


def _launches(N, Q, topk, ctas):
    plan = bg.bergson_debug_score_plan(N, K, Q, topk, ctas)
    launches = bg.bergson_debug_score_launches(N, K, Q, topk, ctas)
    assert len(plan) == len(launches)
    return list(zip(plan, launches))


def check(N, Q, topk, ctas):
    wide = False
    for p, l in _launches(N, Q, topk, ctas):
        assert (l["rows"], l["n_qg"]) == (p["rows"], p["n_qg"])
        # tiles cover the rows in steps one MMA takes (N of 16 at M = 128, of 32 at the pairs'
        # M = 256), and no CTA has one round more than
        # with tiles of 256 rows
        per_group = (min(ctas, 160) & (~1 if p["pair"] else ~0)) // l["n_qg"]
        assert 64 <= l["bn"] <= 256 and l["bn"] % (32 if p["pair"] else 16) == 0
        assert l["n_tiles"] == -(-l["rows"] // l["bn"])
        assert -(-l["n_tiles"] // per_group) <= -(-l["rows"] // (256 * per_group))
        assert 1 <= l["cpg"] <= min(l["n_tiles"], per_group)
        assert l["grid"] == l["n_qg"] * l["cpg"] <= min(ctas, 160)
        # the bound: at least topk first-tile rows lie at or above it
        j, r = l["bound_j"], l["bound_r"]
        assert (j > 0) == (r > 0)
        if j:
            assert j <= 32 and j * r >= topk and r <= l["cpg"]
            # the published words' room, which a wider launch leaves full of list keys
            assert l["grid"] <= 152 and not wide
        wide = wide or l["grid"] > 152


@pytest.mark.parametrize("N,Q,topk,ctas", SIZES)
def test_launches(N, Q, topk, ctas):
    check(N, Q, topk, ctas)


def test_random_launches():
    for size in _random_sizes():
        check(*size)


def test_a_wide_launch_leaves_no_bound_to_the_next():
    # 160 CTAs: 160 query groups, then 18 (8 CTAs each) or 38 (4), whose words would fit
    for groups in (17, 18, 38):
        first, last = bg.bergson_debug_score_launches(9_000, K, 256 * (160 + groups), 10, 160)
        assert first["grid"] == 160 and last["n_qg"] == groups + groups % 2
        assert last["bound_j"] == 0


def test_small_search_is_spread_over_the_sms():
    l, = bg.bergson_debug_score_launches(20_011, 3072, 3, 10, 152)
    assert (l["bn"], l["n_tiles"], l["cpg"], l["grid"]) == (144, 139, 139, 139)
    assert (l["bound_j"], l["bound_r"]) == (1, 10)
