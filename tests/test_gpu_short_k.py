"""Products with a short inner dimension run on 128 x 128 tiles while these are
one wave, longer ones on pairs of CTAs. Zero columns of A and rows of B add zero
digits, so the same product with its inner dimension padded past the rule's line
gives the same integers and the same bits. Sizes on both sides of a tile, of the
wave (19 x 8 tiles, 20 x 8) and of the line (tiles of 256 x 256 times K = 4096)."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,s", [("int8", 7), ("bf16", 6), ("e4m3", 8)])
@pytest.mark.parametrize("m,n,k", [(1000, 333, 257), (1281, 1279, 100), (1793, 129, 1), (2432, 1024, 64),
                                   (2433, 1024, 64), (1024, 1024, 256), (1024, 1024, 257)])
def test_equal_to_the_product_padded_with_zeros(dmp, mode, s, m, n, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(m + n + k)
    A = torch.randn((m, k), generator=g, device="cuda", dtype=torch.float64)
    B = torch.randn((k, n), generator=g, device="cuda", dtype=torch.float64)
    pad = 2048
    A2 = torch.zeros((m, pad), device="cuda", dtype=torch.float64)
    B2 = torch.zeros((pad, n), device="cuda", dtype=torch.float64)
    A2[:, :k], B2[:k] = A, B
    assert torch.equal(dmp.ozaki_gemm(A, B, mode, s), dmp.ozaki_gemm(A2, B2, mode, s))
