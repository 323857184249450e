"""Products of more than 65536 row or column blocks (256 rows or columns each on
pairs of CTAs, 128 rows on single ones): the block index needs more than 16 bits.
The operand repeats a short one, so every part of the result is the short
product's, bit for bit (rows are scaled and split one by one)."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pairing,tall,parts", [(True, True, 16800), (False, True, 8400), (True, False, 16800)])
def test_every_block_is_written(dmp, pairing, tall, parts):
    short, k, other, s = 1000, 64, 64, 4
    g = torch.Generator(device="cuda")
    g.manual_seed(parts)
    A = torch.randn((short, k), generator=g, device="cuda", dtype=torch.float64)
    B = torch.randn((k, other), generator=g, device="cuda", dtype=torch.float64)
    prev = dmp.set_tc_pairing(pairing)
    try:
        if tall:
            want = dmp.ozaki_gemm(A, B, "int8", s, "tc")
            C = torch.full((parts * short, other), float("nan"), dtype=torch.float64, device="cuda")
            dmp.ozaki_gemm(A.repeat(parts, 1), B, "int8", s, "tc", C=C)
            got = C.view(parts, short, other)
        else:
            want = dmp.ozaki_gemm(B.t().contiguous(), A.t().contiguous(), "int8", s, "tc")
            C = torch.full((other, parts * short), float("nan"), dtype=torch.float64, device="cuda")
            dmp.ozaki_gemm(B.t().contiguous(), A.t().contiguous().repeat(1, parts), "int8", s, "tc", C=C)
            got = C.view(other, parts, short).transpose(0, 1)
        assert bool((got == want).all())
    finally:
        dmp.set_tc_pairing(prev)
        del C, got
        torch.cuda.empty_cache()
