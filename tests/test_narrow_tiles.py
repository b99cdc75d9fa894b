"""Products of few tiles run on narrower tensor-core tiles (32, 64 or 128
columns instead of 256).  An output's operations do not depend on the tile, so
every bit equals the same output's inside a product of more tiles than SMs at
128 columns, which takes the 256-wide ones."""
import pytest
import torch

import paper_1801_04723_gb300 as spin

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k", [(1, 1, 64), (127, 31, 8), (128, 32, 65), (129, 33, 200), (1000, 500, 500),
                                   (640, 960, 96), (640, 992, 96), (1024, 1024, 128), (1280, 1280, 72),
                                   (1536, 1536, 1024), (1600, 1600, 64)])
@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-1.0, 1.0)])
def test_narrow_tiles_equal_wide_tiles_bit_by_bit(m, n, k, alpha, beta):
    g = torch.Generator(device="cuda")
    g.manual_seed(m * 1000003 + n * 1009 + k)
    M, N = 2048, 2560
    a = torch.randn(M, k, dtype=torch.float64, device="cuda", generator=g)
    b = torch.randn(k, N, dtype=torch.float64, device="cuda", generator=g)
    c = torch.randn(M, N, dtype=torch.float64, device="cuda", generator=g)
    wide = spin.gemm_bf16x3(a, b, alpha=alpha, beta=beta, C=c if beta else None)
    narrow = spin.gemm_bf16x3(a[:m], b[:, :n], alpha=alpha, beta=beta, C=c[:m, :n] if beta else None)
    assert torch.equal(narrow, wide[:m, :n])
