"""The allocation-free product at inner dimensions whose schedule nearly fills its
16 KB: the bits of the regular entry point; beyond, a refusal."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2509_23565_gb300 import inputs
from paper_2509_23565_gb300.binding import ColMajor, load

pytestmark = pytest.mark.gpu


def _noalloc(A, B, C, s):
    fn = load().emul_dgemm_noalloc
    fn.restype = ctypes.c_int
    vp, ci, cd = ctypes.c_void_p, ctypes.c_int, ctypes.c_double
    fn.argtypes = [vp, ci, ci, ci, cd, vp, ci, vp, ci, cd, vp, ci, ci]
    return fn(torch.cuda.current_stream().cuda_stream, C.m, C.n, A.n, 1.0, A.ptr, A.ld, B.ptr, B.ld, 0.0, C.ptr, C.ld, s)


@pytest.mark.parametrize("k,s", [(28672, 7), (28704, 7), (59712, 7), (51328, 8), (65536, 6)])
def test_long_k(gpu_lib, k, s):
    A, B = (ColMajor.from_numpy(inputs.log_scaled(r, c, 2, seed=k)) for r, c in ((4, k), (k, 5)))
    got, want = ColMajor.empty(4, 5), ColMajor.empty(4, 5)
    assert _noalloc(A, B, got, s) == 0
    gpu_lib.dgemm(A, B, want, s)
    gpu_lib.sync_status()
    assert np.array_equal(got.numpy(), want.numpy()) and got.numpy().any()


def test_schedule_beyond_its_room(gpu_lib):
    A, B, C = ColMajor.empty(2, 65536), ColMajor.empty(65536, 2), ColMajor.empty(2, 2)
    assert _noalloc(A, B, C, 8) == -3
