"""Batches whose systems run on different kernels (fast factorization, general
one, systems handed from the second to the first when their refinement stalls):
each solution is the one that the system alone has."""
import numpy as np
import pytest
import torch

from paper_2509_23565_gb300 import inputs
from paper_2509_23565_gb300.binding import ColMajor

pytestmark = pytest.mark.gpu


def _solve(gpu_lib, As, bs, **kw):
    xs = [ColMajor.from_numpy(b) for b in bs]
    info, berr, iters = gpu_lib.dgesv_batched_ir([ColMajor.from_numpy(A, ld=A.shape[0] + 1) for A in As], xs, **kw)
    torch.cuda.synchronize()
    return [x.numpy()[:, 0] for x in xs], info.cpu().numpy(), berr.cpu().numpy(), iters.cpu().numpy()


def _check_alone(gpu_lib, As, bs, **kw):
    xs, info, berr, iters = _solve(gpu_lib, As, bs, **kw)
    for i, (A, b) in enumerate(zip(As, bs)):
        x, inf, be, it = _solve(gpu_lib, [A], [b], **kw)
        assert np.array_equal(xs[i], x[0]) and (info[i], berr[i], iters[i]) == (inf[0], be[0], it[0]), A.shape[0]
    return xs, berr, iters


@pytest.mark.parametrize("sizes", [(1100, 50, 1025, 300, 64, 1024), (64, 1026), (1025,) * 3 + (40,) * 200, (30, 1030) * 80])
def test_sizes_on_both_sides(gpu_lib, sizes):
    kinds = sorted(set(sizes))
    mats = {n: inputs.uniform(n, n, seed=n) + np.eye(n) for n in kinds}
    vecs = {n: inputs.vector(n, seed=n + 1) for n in kinds}
    xs, info, berr, _ = _solve(gpu_lib, [mats[n] for n in sizes], [vecs[n] for n in sizes], slices=3, nb=32)
    assert not info.any() and (berr <= 1.0).all()
    alone = {n: _solve(gpu_lib, [mats[n]], [vecs[n]], slices=3, nb=32)[0][0] for n in kinds}
    for n, x in zip(sizes, xs):
        assert np.array_equal(x, alone[n])


@pytest.mark.parametrize("slices,nb", [(2, 32), (2, 16), (5, 32), (2, 64), (3, 32)])
def test_stalled_systems(gpu_lib, slices, nb):
    """Systems of condition 1e5 among ordinary ones: 2 slices (14 bits) are too coarse to
    refine with, so these are refactored with 8 slices after eight steps."""
    As, bs = [], []
    for i, n in enumerate((33, 100, 64, 257, 40, 300)):
        As.append(inputs.spd(n, 1e5, seed=n) if i % 2 else inputs.uniform(n, n, seed=n) + 2 * np.eye(n))
        bs.append(inputs.vector(n, seed=n + 1))
    _, berr, iters = _check_alone(gpu_lib, As, bs, slices=slices, nb=nb, max_iter=40)
    if slices == 2:
        assert (iters[1::2] > 8).all()
    assert (berr <= 1.0).all()
