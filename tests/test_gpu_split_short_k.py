"""Slicing around k = 64 and 32768 rows, where blocks change from 8 rows to 32, bit
for bit against the oracle: both storage orders, ragged rows, rows of zeros and
subnormals."""
import numpy as np
import pytest

from oracle import split
from paper_2509_23565_gb300 import inputs
from paper_2509_23565_gb300.binding import ColMajor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 7, 8, 33, 32767, 32768, 32769, 32799])
@pytest.mark.parametrize("k", [1, 8, 9, 64, 65])
@pytest.mark.parametrize("s", [1, 7, 8])
def test_split(gpu_lib, rows, k, s):
    A = inputs.log_scaled(rows, k, 6, seed=rows + k)
    A[rows // 2] = 0.0
    A[rows - 1] *= 2.0 ** -1060                   # subnormals
    e_ref, S_ref = split.split_rows(A, s)
    for X, by in ((ColMajor.from_numpy(A, ld=rows + 3), "rows"), (ColMajor.from_numpy(A.T, ld=k + 1), "cols")):
        exps, sl = gpu_lib.split(X, s, by=by)
        assert np.array_equal(exps.cpu().numpy(), e_ref)
        got = (sl.cpu().numpy().astype(np.int32) << 16).view(np.float32).astype(np.int64)
        assert np.array_equal(got, S_ref.astype(np.int64))
