"""Products of few 16 x 16 tiles run on 8 x 16 or 8 x 8 ones, one output per thread.
An output's operations do not depend on the tile, so every bit equals the same
output's inside a product large enough for the wide tiles."""
import pytest
import torch

import paper_1801_04723_gb300 as spin

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (7, 15, 16), (8, 16, 17), (9, 17, 33), (24, 300, 40), (64, 64, 64),
                                   (5, 2000, 31), (100, 128, 129), (128, 128, 128), (200, 200, 200),
                                   (250, 257, 64), (301, 299, 48), (512, 512, 33)])
@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-1.0, 1.0), (-1.0, 0.0)])
def test_small_tiles_equal_wide_tiles_bit_by_bit(m, n, k, alpha, beta):
    g = torch.Generator(device="cuda")
    g.manual_seed(m * 1000003 + n * 1009 + k)
    M, N = max(m, 1536), max(n, 1536)
    a = torch.randn(M, k, dtype=torch.float64, device="cuda", generator=g)
    b = torch.randn(k, N, dtype=torch.float64, device="cuda", generator=g)
    c = torch.randn(M, N, dtype=torch.float64, device="cuda", generator=g)
    wide = spin.gemm_f64(a, b, alpha=alpha, beta=beta, C=c if beta else None)
    small = spin.gemm_f64(a[:m], b[:, :n], alpha=alpha, beta=beta,
                          C=c[:m, :n] if beta else None)
    assert torch.equal(small, wide[:m, :n])
