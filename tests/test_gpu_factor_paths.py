"""The factorization and solve kernels at the edges of their ranges.

Where two kernels share an operation, the same matrix goes through both and the
results must agree bit for bit: A embedded as diag(A, I) in a larger matrix
reaches the kernel of the larger size, while the added zero rows and columns
change no pivot, scale, digit or sum of A's entries.  Where there is one kernel
only, the factors are integers chosen so that every operation is exact.
"""
import numpy as np
import pytest
import torch

from paper_2509_23565_gb300 import inputs
from paper_2509_23565_gb300.binding import ColMajor

pytestmark = pytest.mark.gpu


def _embed(A, n):
    M = np.eye(n)
    M[:A.shape[0], :A.shape[0]] = A
    return M


def _signs(n, seed):
    """Entries +-1: every pivot search meets ties."""
    return np.where(np.random.default_rng(seed).random((n, n)) < 0.5, -1.0, 1.0)


def _integer_factors(n, seed):
    """Unit lower L and upper U of integers whose block inverses and products are
    exact: the entries off the diagonal stand in even rows and odd columns, so
    (L - I)^2 = 0, and U's diagonal holds powers of two."""
    rng = np.random.default_rng(seed)
    even, odd = (np.arange(n) % 2 == 0)[:, None], (np.arange(n) % 2 == 1)[None, :]
    N = np.where(even & odd, rng.integers(-3, 4, (n, n)), 0).astype(np.float64)
    d = np.exp2(rng.integers(0, 3, n)) * np.where(rng.random(n) < 0.5, -1.0, 1.0)
    return np.tril(N, -1) + np.eye(n), np.triu(N, 1) + np.diag(d)


# ---------------------------------------------------------------- batched factorization
@pytest.mark.parametrize("nb", [16, 32])
@pytest.mark.parametrize("slices", [3, 4, 8])
def test_batched_small_and_large_paths_agree(gpu_lib, nb, slices):
    """The factorization in shared memory (n <= 1024) against the one in global
    memory, which the embedded system takes: the first solutions are equal."""
    As = [inputs.uniform(n, n, seed=n) for n in (1, 2, 15, 16, 17, 31, 32, 33, 47, 48, 49, 64, 65, 100, 257)]
    As += [inputs.log_scaled(n, n, 4, seed=n) for n in (40, 129)] + [_signs(n, n) for n in (50, 96)]
    if nb == 32 or slices == 3:
        As += [inputs.uniform(n, n, seed=n) for n in (511, 512, 513, 1023, 1024)]
    bs = [inputs.vector(A.shape[0], seed=1) for A in As]
    big = 1040
    da = [ColMajor.from_numpy(A, ld=A.shape[0] + i % 3) for i, A in enumerate(As)]
    db = [ColMajor.from_numpy(b) for b in bs]
    ea = [ColMajor.from_numpy(_embed(A, big)) for A in As]
    eb = [ColMajor.from_numpy(np.concatenate([b, np.zeros(big - b.size)])) for b in bs]
    info, _, iters = gpu_lib.dgesv_batched_ir(da, db, max_iter=0, slices=slices, nb=nb)
    einfo, _, _ = gpu_lib.dgesv_batched_ir(ea, eb, max_iter=0, slices=slices, nb=nb)
    gpu_lib.sync_status()
    assert torch.equal(info, einfo) and int(iters.max()) == 0
    for A, b, x, y in zip(As, bs, db, eb):
        n = A.shape[0]
        got, want = x.numpy()[:, 0], y.numpy()[:, 0]
        assert np.array_equal(got, want[:n], equal_nan=True), n
        assert not want[n:].any()


# ---------------------------------------------------------------- panel leaves
@pytest.mark.parametrize("n", [1, 2, 31, 32, 57, 63, 64, 65, 257, 511, 513, 1025, 2047, 2048])
@pytest.mark.parametrize("kind", ["uniform", "signs", "zero column"])
def test_lu_leaves_agree(gpu_lib, n, kind):
    """Leaves of one cluster (at most 2048 rows) against those that exchange
    through global memory, which the embedded matrix's panels take.  (The last
    panels' widths are such that both matrices' recursions split them alike.)"""
    A = _signs(n, n) if kind == "signs" else inputs.uniform(n, n, seed=n)
    if kind == "zero column":
        A[:, n // 2] = 0.0
    big = 2048 + n + 64
    dA, dE = ColMajor.from_numpy(A, ld=n + 1), ColMajor.from_numpy(_embed(A, big))
    ipiv, info = gpu_lib.dgetrf(dA, nb=64, slices=7)
    eipiv, einfo = gpu_lib.dgetrf(dE, nb=64, slices=7)
    gpu_lib.sync_status()
    assert torch.equal(info, einfo)
    assert torch.equal(ipiv, eipiv[:n])
    assert np.array_equal(dA.numpy(), dE.numpy()[:n, :n], equal_nan=True)


# ---------------------------------------------------------------- solves
@pytest.mark.parametrize("n", [1, 2, 31, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 385, 1000])
@pytest.mark.parametrize("nrhs", [1, 2])
def test_solves_exact(gpu_lib, n, nrhs):
    """LU solves with any interchanges, rows above the current one included."""
    L, U = _integer_factors(n, n)
    rng = np.random.default_rng(n + 1)
    X = rng.integers(-8, 9, (n, nrhs)).astype(np.float64)
    piv = rng.integers(1, n + 1, n).astype(np.int32)
    B = L @ (U @ X)                      # integers far below 2^53
    for k in reversed(range(n)):
        p = piv[k] - 1
        B[[k, p]] = B[[p, k]]
    dB = ColMajor.from_numpy(B, ld=n + 1)
    gpu_lib.dgetrs(ColMajor.from_numpy(np.tril(L, -1) + U, ld=n + 2), torch.from_numpy(piv).cuda(), dB)
    gpu_lib.sync_status()
    assert np.array_equal(dB.numpy(), X)


# ---------------------------------------------------------------- Cholesky
@pytest.mark.parametrize("n,nb", [(1, 32), (2, 32), (31, 32), (32, 32), (33, 64), (63, 64), (65, 64), (97, 128),
                                  (129, 48), (200, 96)])
def test_cholesky_blocks(gpu_lib, n, nb):
    """Ragged leaves, panels and blocks.  Within a diagonal block |A - L L^T| <=
    (n + 16) u |L| |L|^T componentwise: n + 1 from the substitutions and sums,
    the rest for the reciprocal root (2 ulp) and the reciprocals.  The rows below
    are a product with the block's inverse, whose error is normwise: up to
    cond(L) = 10 times u per term, of the two rows' largest entries."""
    A = inputs.spd(n, 100.0, seed=n)
    dA = ColMajor.from_numpy(A, ld=n + 1)
    info = gpu_lib.dpotrf(dA, nb=nb, slices=8)
    gpu_lib.sync_status()
    assert int(info.item()) == 0
    L = np.tril(dA.numpy()).astype(np.longdouble)
    scale = np.abs(L).max(axis=1)
    blocks = 10 * n * np.outer(scale, scale) if n > nb else 0.0
    bound = 2.0 ** -53 * ((n + 16) * (np.abs(L) @ np.abs(L).T) + blocks)
    assert (np.abs(np.tril(A - L @ L.T)) <= bound).all()


@pytest.mark.parametrize("at", [0, 1, 7, 8, 31, 32, 33, 63, 64, 69])
def test_cholesky_failing_pivot(gpu_lib, at):
    A = np.eye(70) * 4.0
    A[at, at] = -1.0
    info = gpu_lib.dpotrf(ColMajor.from_numpy(A), nb=64, slices=7)
    assert int(info.item()) == at + 1


def test_cholesky_beside_other_work(gpu_lib):
    """The diagonal blocks' chain on SMs shared with another stream's kernels,
    which delay its warps against each other: the same bits as alone."""
    A = inputs.spd(512, 100.0, seed=3)
    side = torch.cuda.Stream()
    x = torch.rand((1024, 1024), dtype=torch.float64, device="cuda")
    want = None
    for _ in range(8):
        dA = ColMajor.from_numpy(A)
        torch.cuda.synchronize()
        if want is not None:
            with torch.cuda.stream(side):
                for _ in range(100):
                    x.sin_()
        info = gpu_lib.dpotrf(dA, nb=256, slices=7)
        torch.cuda.synchronize()
        assert int(info.item()) == 0
        got = dA.numpy()
        want = got if want is None else want
        assert np.array_equal(got, want)


@pytest.mark.parametrize("n,nb,k", [(6100, 256, 2816), (5000, 128, 2944), (7000, 512, 3072)])
def test_cholesky_ahead_agrees(gpu_lib, n, nb, k):
    """Diagonal blocks factored beside the update (more than 3072 rows right of
    the next block) against the leading submatrix, which has fewer: the leading
    columns' blocks, and so their bits, are the same."""
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    M = torch.rand((n, n), generator=g, dtype=torch.float64, device="cuda")
    M = M + M.T + 2.0 * n * torch.eye(n, dtype=torch.float64, device="cuda")
    small = ColMajor(M[:k, :k].clone(), k, k)
    big = ColMajor(M, n, n)
    info, sinfo = gpu_lib.dpotrf(big, nb=nb, slices=7), gpu_lib.dpotrf(small, nb=nb, slices=7)
    gpu_lib.sync_status()
    assert int(info.item()) == 0 and int(sinfo.item()) == 0
    assert torch.equal(big.store[:k, :k], small.store)


# ---------------------------------------------------------------- no pivoting
@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 31, 32, 33, 63, 64, 65, 80, 127, 129, 200])
@pytest.mark.parametrize("nb", [32, 64, 128])
def test_nopiv_leaves_exact(gpu_lib, n, nb):
    L, U = _integer_factors(n, 7 * n)
    dA = ColMajor.from_numpy(L @ U, ld=n + 1)
    _, info = gpu_lib.dgetrf_nopiv(dA, nb=nb, slices=7)
    gpu_lib.sync_status()
    assert int(info.item()) == 0
    assert np.array_equal(dA.numpy(), np.tril(L, -1) + U)
