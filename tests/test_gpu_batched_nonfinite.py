"""Batched systems that hold NaN, Inf or entries beyond FP32, in both
factorizations: the call returns, and the systems beside them are solved as if
alone."""
import numpy as np
import pytest
import torch

from paper_2509_23565_gb300 import inputs
from paper_2509_23565_gb300.binding import ColMajor

pytestmark = pytest.mark.gpu


def _bad(n, what):
    A = inputs.uniform(n, n, seed=n)
    if what == "nan entry":
        A[n // 2, n // 3] = np.nan
    elif what == "nan column":
        A[:, n // 3] = np.nan
    elif what == "nan first column":
        A[:, 0] = np.nan
    elif what == "nan everywhere":
        A[:] = np.nan
    elif what == "inf entry":
        A[n // 2, n // 3] = np.inf
    else:
        A[n // 2, :] *= 1e300
    return A


@pytest.mark.parametrize("n,nb,slices", [(40, 32, 3), (40, 16, 8), (40, 64, 3), (40, 32, 5), (1, 64, 2), (33, 64, 8),
                                         (1040, 32, 3)])
@pytest.mark.parametrize("what", ["nan entry", "nan column", "nan first column", "nan everywhere", "inf entry",
                                  "beyond fp32"])
def test_no_pivot_candidate(gpu_lib, n, nb, slices, what):
    """A column of the working copy with NaN in every row has no pivot candidate:
    its row stays where it is.  (nb = 64, 5 slices and n > 1024 take the
    factorization in global memory.)"""
    good = inputs.uniform(50, 50, seed=1)
    b = inputs.vector(50, seed=2)
    alone, beside = ColMajor.from_numpy(b), ColMajor.from_numpy(b)
    gpu_lib.dgesv_batched_ir([ColMajor.from_numpy(good)], [alone], nb=nb, slices=slices)
    bx = ColMajor.from_numpy(inputs.vector(n, seed=3))
    info, berr, _ = gpu_lib.dgesv_batched_ir([ColMajor.from_numpy(_bad(n, what)), ColMajor.from_numpy(good)],
                                             [bx, beside], nb=nb, slices=slices)
    torch.cuda.synchronize()
    assert np.array_equal(beside.numpy(), alone.numpy())
    assert int(info[1].item()) == 0 and float(berr[1].item()) <= 1.0


@pytest.mark.parametrize("n,nb,slices", [(40, 32, 3), (100, 64, 3), (1040, 32, 3), (700, 16, 4)])
def test_nan_solution_has_no_backward_error(gpu_lib, n, nb, slices):
    """NaN in the top right corner of a triangular matrix reaches the first entries
    of x only, and through them every residual: the backward error is NaN, not
    that of the finite entries."""
    A = np.triu(inputs.uniform(n, n, seed=n)) / n + 4.0 * np.eye(n)
    A[0, n - 1] = np.nan
    x = ColMajor.from_numpy(inputs.vector(n, seed=3))
    _, berr, _ = gpu_lib.dgesv_batched_ir([ColMajor.from_numpy(A)], [x], nb=nb, slices=slices)
    torch.cuda.synchronize()
    assert np.isnan(x.numpy()[0, 0]) and np.isfinite(x.numpy()[n - 1, 0])
    assert np.isnan(float(berr[0].item()))
