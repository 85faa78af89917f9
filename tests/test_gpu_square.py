"""Square fp32-accurate products (Fisher fit, Newton-Schulz) at tile edges.

Sizes straddle the 128- and 256-row tiles of both kernels, the 64-column stages
and the change from 32- to 64-column accumulation chains, with columns of very
different scale, zero columns and an outlying example, against fp64.
"""
import numpy as np
import pytest
import torch

import paper_2606_11660_gb300 as bg
from oracle import bergson_oracle as orc
from paper_2606_11660_gb300 import workloads as wl
from tests._util import np32

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _fit(x, pad=0):
    n, K = x.shape
    buf = torch.zeros((n, K + pad), device=DEV)
    buf[:, :K] = x.to(DEV)
    R = torch.full((K, K + pad), float("nan"), device=DEV)
    ws = bg.workspace_tensor(bg.bergson_fisher_fit_workspace(n, K), DEV)
    bg.bergson_fisher_fit(buf, n, K, R, ws)
    assert bg.bergson_sync_status() == bg.BERGSON_OK, bg.bergson_last_error()
    return R[:, :K]


@pytest.mark.parametrize("n,K,pad", [(1, 4, 0), (7, 12, 4), (64, 128, 0), (65, 132, 8),
                                     (300, 252, 0), (257, 260, 0), (130, 516, 4), (1025, 1028, 0),
                                     (70, 3076, 0), (513, 3332, 4)])       # 256-wide tiles
def test_fit_at_tile_edges(n, K, pad):
    g = wl.generator(n + K, "cpu")
    x = torch.randn((n, K), generator=g) * torch.logspace(-4, 4, K)
    x[n // 2] *= 2.0 ** 12                    # one example far above the rest
    x[:, K // 2] = 0.0
    R = np32(_fit(x, pad)).astype(np.float64)
    assert np.array_equal(R, R.T)
    want = orc.fisher_fit(x.numpy())
    # per entry, against the Cauchy-Schwarz scale (above chains of 24 sums and n / 32 sums of
    # chains, n / 64 from 513 on): both operands' 2^-23, a chain of at most 48
    # truncating sums of 2^-23, and n / 256 fp32 sums of chains
    d = np.sqrt(np.diag(want))
    err = np.abs(R - want) / np.maximum(np.outer(d, d), 1e-300)
    assert err.max() <= (2 + 48 + (n // 256 + 2)) * 2.0 ** -23, err.max()


def test_fit_keeps_infinities_and_nan_in_their_rows():
    g = wl.generator(3, "cpu")
    x = torch.randn((70, 136), generator=g)
    x[5, 7] = float("inf")
    x[9, 100] = float("nan")
    R = np32(_fit(x))
    bad = np.zeros(136, bool)
    bad[[7, 100]] = True
    assert np.isfinite(R[~bad][:, ~bad]).all()
    assert not np.isfinite(R[bad]).any() and not np.isfinite(R[:, bad]).any()


def test_fit_keeps_small_entries_of_a_column_with_an_outlier():
    # example 5 is 2^36 above the rest, in the even columns only: beside it, R's entries of an even
    # and an odd column are sums of entries 2^-36 of the column's largest
    g = wl.generator(4, "cpu")
    n, K = 300, 260
    x = torch.randn((n, K), generator=g)
    x[5] *= 2.0 ** 36
    x[5, 1::2] = 0.0
    R = np32(_fit(x)).astype(np.float64)[0::2, 1::2]
    xd = x.numpy().astype(np.float64)
    want = (xd[:, 0::2].T @ xd[:, 1::2]) / n
    scale = np.abs(xd[:, 0::2]).T @ np.abs(xd[:, 1::2]) / n
    # both operands' 2^-24, chains of at most 2 + 4 truncating sums, n / 32 fp32 sums of chains
    assert (np.abs(R - want) / scale).max() <= (2 + 6 + n / 32) * 2.0 ** -23


def _power(R, damping, iters=30):
    K = R.shape[0]
    M = torch.full((K, K), float("nan"), device=DEV)
    ws = bg.workspace_tensor(bg.bergson_fisher_preconditioner_workspace(K), DEV)
    bg.bergson_fisher_preconditioner(R.to(DEV), None, K, 1.0, damping, bg.BERGSON_FISHER_INV_SQRT,
                                     iters, M, ws)
    assert bg.bergson_sync_status() == bg.BERGSON_OK, bg.bergson_last_error()
    want = orc.fisher_power(orc.fisher_mix(R.numpy().astype(np.float64), None, 1.0, damping), -0.5)
    return np32(M).astype(np.float64), want


def test_power_keeps_entries_small_beside_the_diagonal():
    # columns of R spread over e^+-8: half of M's entries lie below 1e-6 of sqrt(M_ii M_jj)
    g = wl.generator(40, "cpu")
    K = 256
    x = torch.randn((3 * K, K), generator=g).double() * torch.exp(
        4 * torch.randn((1, K), generator=g).double())
    M, want = _power((x.T @ x / (3 * K)).float(), 0.1)
    assert np.median(np.abs(M - want) / np.abs(want)) < 1e-3     # 7e-5 with tf32 parts


@pytest.mark.parametrize("K", [128, 256, 512])
def test_power_error_at_small_K(K):
    g = wl.generator(41 + K, "cpu")
    x = torch.randn((3 * K, K), generator=g)
    M, want = _power((x.T @ x / (3 * K)).float(), 0.1)
    # a product is off by at most 4 truncations of 2^-23 (a chain's two and the terms before them),
    # an update by three products', and sqrt(cond R) = 3.7 is the iteration's amplification
    assert np.linalg.norm(M - want) / np.linalg.norm(want) < 4 * 3 * 3.7 * 2.0 ** -23


@pytest.mark.parametrize("K", [4, 60, 132, 260, 516, 1028, 2052])    # from 1028: 256-wide tiles, ragged
@pytest.mark.parametrize("power", [bg.BERGSON_FISHER_INV_SQRT, bg.BERGSON_FISHER_INV])
def test_power_at_tile_edges(K, power):
    g = wl.generator(K, "cpu")
    x1 = torch.randn((2 * K, K), generator=g) * torch.linspace(0.5, 2.0, K)
    x2 = torch.randn((K + 3, K), generator=g)
    R1, R2 = orc.fisher_fit(x1.numpy()), orc.fisher_fit(x2.numpy())
    M = torch.full((K, K + 4), float("nan"), device=DEV)
    ws = bg.workspace_tensor(bg.bergson_fisher_preconditioner_workspace(K), DEV)
    t1, t2 = (torch.tensor(r, dtype=torch.float32, device=DEV) for r in (R1, R2))
    done, res = bg.bergson_fisher_preconditioner_tol(t1, t2, K, 0.25, 0.1, power, 40, 2e-5, M, ws)
    assert bg.bergson_sync_status() == bg.BERGSON_OK, bg.bergson_last_error()
    assert done < 40 and res[-1] <= 2e-5
    p = -0.5 if power == bg.BERGSON_FISHER_INV_SQRT else -1.0
    want = orc.fisher_power(orc.fisher_mix(R1, R2, 0.25, 0.1), p)
    got = np32(M)[:, :K].astype(np.float64)
    # the residual bounds ||M R M - I||; the inverse doubles it, the condition number is below 100
    assert np.linalg.norm(got - want) / np.linalg.norm(want) < 1e-3


@pytest.mark.parametrize("power", [bg.BERGSON_FISHER_INV_SQRT, bg.BERGSON_FISHER_INV])
def test_power_that_starts_converged(power):
    # R = I at K = 4 has c = 2: a tolerance above the first residual stops at Z = I
    R = torch.eye(4, device=DEV)
    M = torch.full((4, 4), float("nan"), device=DEV)
    ws = bg.workspace_tensor(bg.bergson_fisher_preconditioner_workspace(4), DEV)
    done, res = bg.bergson_fisher_preconditioner_tol(R, None, 4, 1.0, 0.0, power, 10, 0.9, M, ws)
    assert done == 0 and len(res) == 1 and abs(res[0] - 0.5) < 1e-6
    want = 2.0 ** (-0.5 if power == bg.BERGSON_FISHER_INV_SQRT else -1.0)
    np.testing.assert_allclose(np32(M), np.eye(4) * want, rtol=1e-6)


def _r256(n):
    return -(-n // 256) * 256


def _fp16_sizes(n, K):
    """The workspaces of fit and power with operands in two fp16 planes and a scale per row."""
    split = lambda rows, cols: _r256(4 * rows * (-(-cols // 8) * 8)) + _r256(4 * rows)
    part = max(K, (-(-K // 64)) ** 2, 16 * -(-K // 256) * -(-K // 128))
    return (split(K, n) + _r256(4 * K),
            2 * _r256(4 * K * K) + 4 * split(K, K) + _r256(36 * K) + _r256(4 * part) + 512)


@pytest.mark.parametrize("n,K", [(9, 128), (70, 132), (300, 260), (1025, 516), (513, 1028)])
def test_smaller_workspaces(n, K):
    # room for two thirds of the rows: R in two parts; for three splits: the products one by one
    g = wl.generator(n, "cpu")
    x = torch.randn((n, K), generator=g) * torch.logspace(-1, 1, K)
    fit_bytes, power_bytes = _fp16_sizes(n, K)
    assert fit_bytes < bg.bergson_fisher_fit_workspace(n, K)
    assert power_bytes < bg.bergson_fisher_preconditioner_workspace(K)
    R = torch.full((K, K), float("nan"), device=DEV)
    bg.bergson_fisher_fit(x.to(DEV), n, K, R, bg.workspace_tensor(fit_bytes, DEV)[:fit_bytes])
    assert bg.bergson_sync_status() == bg.BERGSON_OK, bg.bergson_last_error()
    want = orc.fisher_fit(x.numpy())
    d = np.sqrt(np.diag(want))
    err = np.abs(np32(R).astype(np.float64) - want) / np.outer(d, d)
    assert err.max() <= (2 + 24 + n / 32 + 2) * 2.0 ** -23 and torch.equal(R, R.T)
    for power in (bg.BERGSON_FISHER_INV_SQRT, bg.BERGSON_FISHER_INV):
        for tol in (0.0, 1e-3):
            out = []
            for size in (bg.bergson_fisher_preconditioner_workspace(K), power_bytes):
                M = torch.full((K, K), float("nan"), device=DEV)
                ws = bg.workspace_tensor(size, DEV)[:size]
                ws.fill_(0x7F)
                out.append((M, bg.bergson_fisher_preconditioner_tol(R, None, K, 1.0, 0.1, power, 12,
                                                                    tol, M, ws)))
                assert bg.bergson_sync_status() == bg.BERGSON_OK, bg.bergson_last_error()
            assert torch.equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]
            assert not torch.isnan(out[0][0]).any()


@pytest.mark.parametrize("K", [8, 604, 1284])
@pytest.mark.parametrize("tol", [0.0, 1e-4])
def test_a_norm_that_overflows_gives_nan(K, tol):
    # ||R||_F^2 > 2^128: no scale to iterate from, and not M = 0
    R = torch.eye(K, device=DEV) * 1e25
    for power in (bg.BERGSON_FISHER_INV_SQRT, bg.BERGSON_FISHER_INV):
        M = torch.zeros((K, K), device=DEV)
        ws = bg.workspace_tensor(bg.bergson_fisher_preconditioner_workspace(K), DEV)
        done, res = bg.bergson_fisher_preconditioner_tol(R, None, K, 1.0, 0.1, power, 5, tol, M, ws)
        assert bg.bergson_sync_status() == bg.BERGSON_OK, bg.bergson_last_error()
        assert torch.isnan(M).all() and done == 5 and np.isnan(res).all()
