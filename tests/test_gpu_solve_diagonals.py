"""Triangular solves over every kind of diagonal: a diagonal matrix's solution is
one division per entry, known exactly."""
import numpy as np
import pytest
import torch

from paper_2509_23565_gb300.binding import ColMajor

pytestmark = pytest.mark.gpu


def _lu_solve(gpu_lib, T, B):
    n = T.shape[0]
    dB = ColMajor.from_numpy(B, ld=n + 1)
    gpu_lib.dgetrs(ColMajor.from_numpy(T, ld=n + 2), torch.arange(1, n + 1, dtype=torch.int32, device="cuda"), dB)
    gpu_lib.sync_status()
    return dB.numpy()


def _chol_solve(gpu_lib, T, B):
    n = T.shape[0]
    dB = ColMajor.from_numpy(B, ld=n + 1)
    gpu_lib.dpotrs(ColMajor.from_numpy(T, ld=n + 2), dB)
    gpu_lib.sync_status()
    return dB.numpy()


def _magnitudes(rng, shape, lo, hi):
    return rng.uniform(1.0, 2.0, shape) * np.exp2(rng.integers(lo, hi, shape)) * rng.choice([-1.0, 1.0], shape)


@pytest.mark.parametrize("n", [1, 32, 127, 128, 300])
@pytest.mark.parametrize("lo,hi", [(-3, 4), (-390, 390), (-499, 499)])
def test_quotients(gpu_lib, n, lo, hi):
    """Several right-hand sides: x = b / d rounded once, by the diagonal's reciprocals
    (|d|, |b| within 2^-400 .. 2^400) and outside them.  One right-hand side:
    x = b RN(1 / d), two roundings."""
    rng = np.random.default_rng(n)
    d, B = _magnitudes(rng, n, lo, hi), _magnitudes(rng, (n, 40), lo, hi)
    B[rng.random(B.shape) < 0.1] = 0.0
    want = B / d[:, None]
    assert np.array_equal(_lu_solve(gpu_lib, np.diag(d), B), want)
    assert np.array_equal(_lu_solve(gpu_lib, np.diag(d), B[:, :1]), B[:, :1] * (1.0 / d)[:, None])
    lo, hi = max(lo, -300), min(hi, 300)             # (b / d) / d stays normal
    d, B = np.abs(_magnitudes(rng, n, lo, hi)), _magnitudes(rng, (n, 2), lo, hi)
    want = B / d[:, None] / d[:, None]
    assert np.array_equal(_chol_solve(gpu_lib, np.diag(d), B), want)


@pytest.mark.parametrize("n", [1, 33, 130, 257])
@pytest.mark.parametrize("nrhs", [1, 2, 5])
@pytest.mark.parametrize("e", [-1074, -1030, -1025, -1022, 1022, 1023])
def test_reciprocals_out_of_range(gpu_lib, n, nrhs, e):
    """Diagonal entries near 2^e, whose reciprocals are infinite or short of bits,
    among ordinary ones: the quotients are ordinary numbers.  A block that holds
    one such entry divides throughout."""
    rng = np.random.default_rng(n + e + 1074)
    X = rng.integers(-8, 9, (n, nrhs)).astype(np.float64)
    small = np.ldexp(1.0, e) * (1.0 if e == -1074 else 1.25)
    d = np.where(rng.random(n) < 0.5, small, 3.0)
    d[0] = d[-1] = small
    if e > 0:
        X /= 16.0                                    # (d X stays finite)
    B = X * d[:, None]                               # exact: few bits
    assert np.array_equal(_lu_solve(gpu_lib, np.diag(d), B), X)
    # the whole triangle at that scale, with a chain through all rows
    if e < 0:
        U = np.triu(rng.integers(-1, 2, (n, n))).astype(np.float64)
        np.fill_diagonal(U, 1.0)
        assert np.array_equal(_lu_solve(gpu_lib, np.ldexp(U, e), np.ldexp(U @ X, e)), X)


@pytest.mark.parametrize("nrhs", [1, 3])
def test_special_diagonals(gpu_lib, nrhs):
    """Zero, infinite and NaN entries in the last row of an upper triangle (the
    first to be solved) and what they make of x there."""
    b = np.array([3.0, -2.0, 0.0])[:nrhs]
    for d in (0.0, np.inf, -np.inf, np.nan):
        with np.errstate(all="ignore"):
            want = b / d
        T = np.diag([2.0, d])
        got = _lu_solve(gpu_lib, T, np.vstack([np.zeros(nrhs), b]))
        assert np.array_equal(got[1], want, equal_nan=True)


@pytest.mark.parametrize("nrhs", [1, 2])
def test_cholesky_factor_of_tiny_scale(gpu_lib, nrhs):
    n = 130
    d = np.full(n, 2.0 ** -1030)
    k = np.random.default_rng(1).integers(-15, 16, (n, nrhs)).astype(np.float64)
    assert np.array_equal(_chol_solve(gpu_lib, np.diag(d), np.ldexp(k, -1070)), np.ldexp(k, 990))
