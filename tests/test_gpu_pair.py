"""The product's CTA-pair variant at the edges of its tiles and schedules, bit
for bit against the oracle (the result is defined exactly: an exact sum, one
rounding): tile remainders in both tile widths, K around the 32-chunk and the
exactness groups, the low bits put aside (8 slices, long K), level sums that
leave the 2^22 range of the quick integer conversion (entries of one sign), and
every update of C."""
import numpy as np
import pytest

from oracle import emulgemm
from paper_2509_23565_gb300 import inputs
from paper_2509_23565_gb300.binding import ColMajor

pytestmark = pytest.mark.gpu


def _check(lib, A, B, s, alpha, beta, seed, ld=0):
    m, n = A.shape[0], B.shape[1]
    C = inputs.uniform(m, n, seed=seed)
    dC = ColMajor.from_numpy(C, ld=m + ld)
    lib.dgemm(ColMajor.from_numpy(A, ld=m + ld), ColMajor.from_numpy(B, ld=B.shape[0] + ld), dC, s, alpha, beta)
    lib.sync_status()
    want = emulgemm.emul_gemm(A, B, s, alpha=alpha, beta=beta, C=C)
    assert np.array_equal(dC.numpy().view(np.int64), want.view(np.int64))


@pytest.mark.parametrize("m,n", [(129, 1), (130, 63), (257, 65), (256, 128), (385, 129)])
@pytest.mark.parametrize("k", [1, 33, 130])
@pytest.mark.parametrize("s", [3, 7, 8])
def test_pair_tiles(gpu_lib, m, n, k, s):
    _check(gpu_lib, inputs.log_scaled(m, k, 2, seed=m + k), inputs.uniform(k, n, seed=n + s), s, -1.0, 1.0, 7, ld=k % 2)


@pytest.mark.parametrize("k", [1024, 1056, 2080])
@pytest.mark.parametrize("s,alpha,beta", [(7, 1.0, 0.0), (8, -1.0, 1.0), (6, 0.5, -2.0), (8, 0.5, -2.0)])
def test_pair_long_k(gpu_lib, k, s, alpha, beta):
    _check(gpu_lib, inputs.uniform(131, k, seed=k), inputs.uniform(k, 21, seed=s), s, alpha, beta, 9)


@pytest.mark.parametrize("s", [4, 7, 8])
@pytest.mark.parametrize("k", [256, 1040])
def test_pair_one_sign(gpu_lib, s, k):
    """Entries in [1/2, 1): every product positive, the level sums near the budget."""
    A, B = inputs.uniform(140, k, seed=3, lo=0.5, hi=1.0), inputs.uniform(k, 18, seed=4, lo=0.5, hi=1.0)
    A[:70] = 1.0 - 2.0 ** -53            # all digits 127
    B[:, :9] = 1.0 - 2.0 ** -53
    _check(gpu_lib, A, B, s, -1.0, 1.0, 11)
    _check(gpu_lib, -A, B, s, 1.0, 0.0, 12)


def test_pair_zero_and_extreme_scales(gpu_lib):
    """Exact zeros, cancellation to zero, results that leave the normal range, infinities."""
    A = inputs.uniform(150, 64, seed=5)
    B = inputs.uniform(64, 70, seed=6)
    A[3] = 0.0
    A[:, 32:] = A[:, :32]
    B[32:, 5] = -B[:32, 5]               # column 5 cancels exactly
    A[10] *= 2.0 ** -1000
    B[:, 7] *= 2.0 ** -70
    A[11] *= 2.0 ** 900
    B[:, 8] *= 2.0 ** 200
    A[12, 1] = np.inf
    for s in (7, 8):
        C = np.zeros((150, 70), order="F")
        dC = ColMajor.from_numpy(C)
        gpu_lib.dgemm(ColMajor.from_numpy(A), ColMajor.from_numpy(B), dC, s, 1.0, 0.0)
        gpu_lib.sync_status()
        rows = np.r_[0:12, 13:150]
        want = emulgemm.emul_gemm(A[rows], B, s)
        got = dC.numpy()
        assert np.array_equal(got[rows].view(np.int64) << 1, want.view(np.int64) << 1)   # the sign of a zero aside
        assert np.isnan(got[12]).all()
