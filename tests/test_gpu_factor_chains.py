"""Leaves and solves on integer factors whose every operation is exact and in
which each step feeds the next: an update that is left out, taken from stale
values or out of order gives another result (which each test asserts of the CPU
variants that do so)."""
import numpy as np
import pytest
import torch

from paper_2509_23565_gb300.binding import ColMajor

pytestmark = pytest.mark.gpu


def _dense(n, seed):
    """Dense unit lower L of -1, 0, 1 and upper U of integers with powers of two on
    the diagonal: elimination of L U and substitution stay in small integers."""
    rng = np.random.default_rng(seed)
    L = np.tril(rng.integers(-1, 2, (n, n)), -1).astype(np.float64) + np.eye(n)
    d = np.exp2(rng.integers(0, 3, n)) * np.where(rng.random(n) < 0.5, -1.0, 1.0)
    return L, np.triu(rng.integers(-3, 4, (n, n)), 1) + np.diag(d)


def _sparse_lower(n, rng):
    """Unit lower triangle of -1, 0, 1: one entry per row at most five left of the
    diagonal (chains through all rows) and a tenth of the entries outside the diagonal
    blocks of 32, so that the inverses of its blocks of 128 stay small."""
    L = np.where(rng.random((n, n)) < 0.1, rng.choice([-1.0, 1.0], (n, n)), 0.0)
    L[np.arange(n)[:, None] // 32 <= np.arange(n) // 32] = 0.0
    L += np.eye(n)
    for i in range(1, n):
        L[i, rng.integers(max(0, i - 5), i)] = rng.choice([-1.0, 1.0])
    return L


def _eliminate(A, update=lambda k, rows, cols: (rows, cols)):
    """Right-looking elimination; `update` gives the part of the trailing matrix
    (rows, columns from k + 1 on) that pivot k's update reaches."""
    A, n = A.copy(), A.shape[0]
    for k in range(n):
        A[k + 1:, k] /= A[k, k]
        rows, cols = update(k, slice(k + 1, n), slice(k + 1, n))
        A[rows, cols] -= np.outer(A[rows, k], A[k, cols])
    return A


def _none(k, rows, cols):
    return slice(0, 0), cols


def _right_half_stale(k, rows, cols):        # columns from 32 on miss the pivots before 32
    return rows, slice(cols.start, 32) if k < 32 else cols


def _within(nb):                             # updates stop at the block's last column
    return lambda k, rows, cols: (rows, slice(cols.start, (k // nb + 1) * nb))


@pytest.mark.parametrize("n", [1, 2, 3, 7, 8, 9, 16, 17, 24, 25, 31, 32, 33, 34, 39, 40, 41, 48, 56, 57, 63, 64])
def test_nopiv_leaf(gpu_lib, n):
    """One leaf of n columns."""
    L, U = _dense(n, n)
    want = np.tril(L, -1) + U
    assert np.array_equal(_eliminate(L @ U), want)
    with np.errstate(all="ignore"):
        for stale in [_none] * (n >= 7) + [_right_half_stale] * (n >= 39):
            assert not np.array_equal(_eliminate(L @ U, stale), want)
    dA = ColMajor.from_numpy(L @ U, ld=n + 1)
    _, info = gpu_lib.dgetrf_nopiv(dA, nb=64, slices=7)
    gpu_lib.sync_status()
    assert int(info.item()) == 0
    assert np.array_equal(dA.numpy(), want)


@pytest.mark.parametrize("n", [65, 80, 127, 129, 200, 333])
@pytest.mark.parametrize("nb", [32, 64, 128])
def test_nopiv_blocks(gpu_lib, n, nb):
    """Several leaves: their inverses, L21, U12 and the Schur updates.  The blocks'
    inverses hold integers below 2^14 (two slices), so the products of three of
    them keep every slice pair that is not zero (p + q <= 8)."""
    rng = np.random.default_rng(1000 * nb + n)
    L, U = _sparse_lower(n, rng), _sparse_lower(n, rng).T * np.where(rng.random(n) < 0.5, -1.0, 1.0)[:, None]
    for d in range(0, n, 128):
        for T in (L, U):
            assert np.abs(np.linalg.inv(T[d:d + 128, d:d + 128])).max() < 2 ** 14
    want = np.tril(L, -1) + U
    assert np.array_equal(_eliminate(L @ U), want)
    with np.errstate(all="ignore"):
        assert not np.array_equal(_eliminate(L @ U, _none), want)
        if n > 65:
            assert not np.array_equal(_eliminate(L @ U, _within(min(nb, 64))), want)
    dA = ColMajor.from_numpy(L @ U, ld=n + 1)
    _, info = gpu_lib.dgetrf_nopiv(dA, nb=nb, slices=7)
    gpu_lib.sync_status()
    assert int(info.item()) == 0
    assert np.array_equal(dA.numpy(), want)


def _forward(L, b, step=1, lag=0):
    """Substitution with unit lower L; with `lag`, a row misses the newest `lag` of the
    steps (of `step` rows) before it."""
    x = b.copy()
    for i in range(L.shape[0]):
        j = max(0, i // step - lag) * step if lag else i
        x[i] -= L[i, :j] @ x[:j]
    return x


@pytest.mark.parametrize("n", [1, 2, 7, 9, 31, 33, 64, 65, 127, 128, 129, 255, 257, 385, 700])
@pytest.mark.parametrize("nrhs", [1, 2, 7])
def test_solves(gpu_lib, n, nrhs):
    """Both substitutions through chains over every 8-row step and 128-row block."""
    L, U = _dense(n, n)
    rng = np.random.default_rng(n + 1)
    X = rng.integers(-8, 9, (n, nrhs)).astype(np.float64)
    Y = U @ X
    B = L @ Y
    assert np.abs(B).max() < 2 ** 40 and np.array_equal(_forward(L, B), Y)
    if n > 2:
        assert not np.array_equal(B - np.tril(L, -1) @ B, Y)               # no chain at all
    if n > 9:
        assert not np.array_equal(_forward(L, B, 8, 1), Y)
    if n > 257:
        assert not np.array_equal(_forward(L, B, 128, 1), Y)
    piv = rng.integers(1, n + 1, n).astype(np.int32)
    P = B.copy()
    for k in reversed(range(n)):
        P[[k, piv[k] - 1]] = P[[piv[k] - 1, k]]
    dB = ColMajor.from_numpy(P, ld=n + 1)
    gpu_lib.dgetrs(ColMajor.from_numpy(np.tril(L, -1) + U, ld=n + 2), torch.from_numpy(piv).cuda(), dB)
    gpu_lib.sync_status()
    assert np.array_equal(dB.numpy(), X)
    # Cholesky: L D with powers of two on the diagonal
    C = L * np.abs(np.diag(U))
    dB = ColMajor.from_numpy(C @ (C.T @ X), ld=n + 1)
    gpu_lib.dpotrs(ColMajor.from_numpy(C, ld=n + 2), dB)
    gpu_lib.sync_status()
    assert np.array_equal(dB.numpy(), X)
