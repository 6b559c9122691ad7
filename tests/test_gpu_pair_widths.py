"""Products on 128-column pair tiles against the same product taken in column
blocks that are narrow enough for 64-column tiles: the same bits."""
import pytest
import torch

from paper_2509_23565_gb300.binding import ColMajor

pytestmark = pytest.mark.gpu


def _entries(m, n, seed, one_sign):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.rand((n, m), generator=g, dtype=torch.float64, device="cuda")
    return x * 0.5 + 0.5 if one_sign else (x - 0.5) * torch.pow(10.0, 4 * torch.rand_like(x) - 2)


@pytest.mark.parametrize("m,n", [(4864, 257), (4900, 300), (2600, 513), (9985, 130), (18000, 65)])
@pytest.mark.parametrize("k,s", [(33, 7), (256, 3), (256, 7), (256, 8), (1056, 7)])
@pytest.mark.parametrize("one_sign", [False, True])
def test_widths_agree(gpu_lib, m, n, k, s, one_sign):
    """(m, n) has more 64-column tiles than CTA pairs; a third of its columns, or 64
    of them, has not."""
    A, B = _entries(m, k, 1, one_sign), _entries(k, n, 2, one_sign)
    C0 = _entries(m, n, 3, False)
    for alpha, beta in [(-1.0, 1.0), (1.0, 0.0), (0.5, -2.0)]:
        C, D = C0.clone(), C0.clone()
        gpu_lib.dgemm(ColMajor(A, m, k), ColMajor(B, k, n), ColMajor(C, m, n), s, alpha, beta)
        w = 64 if n < 200 else (n + 2) // 3 + 63 & ~63
        for c in range(0, n, w):
            e = min(n, c + w)
            gpu_lib.dgemm(ColMajor(A, m, k), ColMajor(B[c:e], k, e - c), ColMajor(D[c:e], m, e - c), s, alpha, beta)
        gpu_lib.sync_status()
        assert torch.equal(C, D)


@pytest.mark.parametrize("k,s", [(100, 8), (300, 8), (1100, 7), (256, 7)])
def test_level_sums_widths_agree(gpu_lib, k, s):
    """Level sums of a product too large for one wave of CTA pairs against those of
    its column blocks."""
    m, n = 2100, 700
    A, B = _entries(m, k, 1, False), _entries(k, n, 2, False)
    whole = gpu_lib.level_sums(ColMajor(A, m, k), ColMajor(B, k, n), s)
    for c in range(0, n, 256):
        e = min(n, c + 256)
        assert torch.equal(whole[:, c:e], gpu_lib.level_sums(ColMajor(A, m, k), ColMajor(B[c:e], k, e - c), s))
