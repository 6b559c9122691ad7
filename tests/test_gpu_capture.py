"""Products recorded into a CUDA graph after other products with the same inner
dimension and slice count: nothing is left to allocate."""
import pytest
import torch

from paper_2509_23565_gb300.binding import ColMajor, Emul

pytestmark = pytest.mark.gpu


def _entries(m, n, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return ColMajor(torch.rand((n, m), generator=g, dtype=torch.float64, device="cuda") - 0.5, m, n)


@pytest.mark.parametrize("k,s", [(256, 7), (300, 8), (2000, 7)])
@pytest.mark.parametrize("first,then", [(700, 100), (100, 700)])
def test_capture_after_another_shape(gpu_lib, k, s, first, then):
    """Products of more than 128 rows and others run on different kernel variants."""
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        e = Emul()
        n = 400
        e.dgemm(_entries(1000, 4 * k, 1), _entries(4 * k, n, 2), _entries(1000, n, 3), s)      # sizes the workspace
        A, B = _entries(then, k, 4), _entries(k, n, 5)
        e.dgemm(_entries(first, k, 6), B, _entries(first, n, 7), s)
        C = _entries(then, n, 8)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            e.dgemm(A, B, C, s)
        graph.replay()
        torch.cuda.synchronize()
        e.sync_status()
    want = ColMajor.empty(then, n)
    gpu_lib.dgemm(A, B, want, s)
    assert torch.equal(C.store, want.store)
