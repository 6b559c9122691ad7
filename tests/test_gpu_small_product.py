"""The one-launch product (short K, few tiles) bit for bit against the oracle at
the edges of its tiles and K halves, for both operand orders, with C inside the
operands' matrix and in place over an operand, where its blocks could read what
another block has written."""
import numpy as np
import pytest
import torch

from oracle import emulgemm
from paper_2509_23565_gb300 import inputs
from paper_2509_23565_gb300.binding import ColMajor

pytestmark = pytest.mark.gpu


def _same(got, want):
    assert np.array_equal(got.view(np.int64), want.view(np.int64))


def _view(M, r, c, m, n):
    """The m x n block at (r, c) of the column-major M (same memory)."""
    V = ColMajor(M.store, m, n)
    V.store = M.store[c:, r:]
    V.ld = M.ld
    return V


@pytest.mark.parametrize("m,n", [(1, 1), (128, 32), (129, 33), (300, 70), (64, 200)])
@pytest.mark.parametrize("k", [1, 16, 17, 32, 33, 64, 65, 100, 128, 129])
@pytest.mark.parametrize("s", [3, 7, 8])
def test_small_shapes(gpu_lib, m, n, k, s):
    A, B, C = inputs.log_scaled(m, k, 3, seed=m + k), inputs.uniform(k, n, seed=n), inputs.uniform(m, n, seed=1)
    for alpha, beta in ((1.0, 0.0), (-1.0, 1.0), (0.5, -2.0)):
        dC = ColMajor.from_numpy(C, ld=m + 1)
        gpu_lib.dgemm(ColMajor.from_numpy(A, ld=m + 2), ColMajor.from_numpy(B), dC, s, alpha, beta)
        gpu_lib.sync_status()
        _same(dC.numpy(), emulgemm.emul_gemm(A, B, s, alpha=alpha, beta=beta, C=C))


@pytest.mark.parametrize("s", [1, 5, 8])
def test_small_one_sign_and_special(gpu_lib, s):
    """Digits of 127 and one sign at the largest K, zeros, subnormals, far scales, infinities."""
    A = np.full((140, 128), 1.0 - 2.0 ** -53)
    B = np.full((128, 40), 1.0 - 2.0 ** -53)
    A[5] = 0.0
    A[6] *= 2.0 ** -1040
    A[7] *= 2.0 ** 1000
    A[8, ::2] *= -1.0
    B[:, 3] *= 2.0 ** 100
    B[:, 4] *= 2.0 ** -60
    A[139, 0] = np.inf
    dC = ColMajor.from_numpy(np.zeros((140, 40)))
    gpu_lib.dgemm(ColMajor.from_numpy(A), ColMajor.from_numpy(B), dC, s)
    gpu_lib.sync_status()
    want = emulgemm.emul_gemm(A[:139], B, s)
    got = dC.numpy()
    assert np.array_equal(got[:139].view(np.int64) << 1, want.view(np.int64) << 1)   # the sign of a zero aside
    assert np.isnan(got[139]).all()


@pytest.mark.parametrize("m,n,k", [(200, 48, 40), (100, 90, 64), (300, 30, 30)])
def test_small_inside_one_matrix(gpu_lib, m, n, k):
    """A21, A12 and A22 of one matrix, as the panel recursion has them."""
    M = inputs.uniform(k + m, k + n, seed=m)
    dM = ColMajor.from_numpy(M)
    gpu_lib.dgemm(_view(dM, k, 0, m, k), _view(dM, 0, k, k, n), _view(dM, k, k, m, n), 7, -1.0, 1.0)
    gpu_lib.sync_status()
    want = M.copy(order="F")
    want[k:, k:] = emulgemm.emul_gemm(M[k:, :k], M[:k, k:], 7, alpha=-1.0, beta=1.0, C=M[k:, k:])
    _same(dM.numpy(), want)


@pytest.mark.parametrize("over,m,n,k", [("B", 128, 200, 128), ("B", 64, 90, 64), ("B", 150, 90, 100), ("B", 100, 40, 128),
                                        ("A", 300, 32, 32), ("A", 300, 64, 64), ("A", 100, 20, 70), ("shift", 90, 50, 60)])
def test_small_in_place(gpu_lib, over, m, n, k):
    """C over an operand (or one row and column off it) gives what separate memory gives."""
    A, B = inputs.uniform(m, k, seed=2), inputs.uniform(k, n, seed=3)
    rows, cols = max(m, k) + 1, max(n, k) + 1
    buf = np.zeros((rows, cols))
    if over == "A":
        buf[:m, :k] = A
    else:
        buf[:k, :n] = B
    dbuf = ColMajor.from_numpy(buf)
    dA = _view(dbuf, 0, 0, m, k) if over == "A" else ColMajor.from_numpy(A)
    dB = ColMajor.from_numpy(B) if over == "A" else _view(dbuf, 0, 0, k, n)
    o = 1 if over == "shift" else 0
    gpu_lib.dgemm(dA, dB, _view(dbuf, o, o, m, n), 6)
    gpu_lib.sync_status()
    torch.cuda.synchronize()
    _same(np.ascontiguousarray(dbuf.numpy()[o:o + m, o:o + n].T).T, emulgemm.emul_gemm(A, B, 6))
