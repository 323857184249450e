"""The output step of the tcgen05 product (ozaki_finish_kernel) and the sharing
of tiles, at the sizes and layouts where they can go wrong: edges of 32-wide
blocks and of tiles, odd leading dimensions and 8-byte aligned outputs (the
element-by-element path), one, two and three group sums per element, results
outside the normal range, and NaN rows. Every result must be the oracle's bits:
the level sums are exact integers and the float64 steps are defined."""

import numpy as np
import pytest
import torch

from oracle import ozaki as oz

pytestmark = pytest.mark.gpu

RULE = {"int8": (7, "trunc"), "bf16": (8, "nearest"), "e4m3": (5, "nearest")}


def _want(A, B, mode, s):
    beta, rounding = RULE[mode]
    return oz.ozaki_gemm(A, B, s, beta, rounding=rounding)


def _into(dmp, A, B, mode, s, pad, shift):
    """ozaki_gemm into a view of leading dimension n + pad that starts `shift`
    elements into its buffer; the elements around the view stay untouched."""
    m, n = A.shape[0], B.shape[1]
    buf = torch.full((m * (n + pad) + shift,), 7.5, dtype=torch.float64, device="cuda")
    C = buf[shift:].view(m, n + pad)[:, :n]
    dmp.ozaki_gemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), mode, s, "tc", C=C)
    if pad:
        assert bool((buf[shift:].view(m, n + pad)[:, n:] == 7.5).all())
    assert bool((buf[:shift] == 7.5).all())
    return C.cpu().numpy()


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (31, 33, 64), (32, 32, 65), (127, 257, 128), (129, 255, 200),
                                   (256, 256, 130), (300, 520, 90)])
@pytest.mark.parametrize("mode,s", [("int8", 5), ("int8", 8), ("bf16", 7), ("e4m3", 9)])
def test_edges_of_blocks_and_tiles(dmp, m, n, k, mode, s):
    rng = np.random.default_rng(m + 10 * n + 100 * k + s)
    A, B = rng.standard_normal((m, k)), rng.standard_normal((k, n))
    assert np.array_equal(_into(dmp, A, B, mode, s, 0, 0), _want(A, B, mode, s))


@pytest.mark.parametrize("pad,shift", [(1, 0), (2, 1), (3, 1), (0, 1)])
@pytest.mark.parametrize("mode,s", [("int8", 5), ("int8", 8)])
def test_layouts_without_16_byte_access(dmp, pad, shift, mode, s):
    rng = np.random.default_rng(pad + 4 * shift + s)
    A, B = rng.standard_normal((100, 96)), rng.standard_normal((96, 70))
    assert np.array_equal(_into(dmp, A, B, mode, s, pad, shift), _want(A, B, mode, s))


@pytest.mark.parametrize("s", [4, 8])
def test_results_outside_the_normal_range(dmp, s):
    """Rows scaled so that products are subnormal, zero or near the largest
    double, in one matrix with ordinary rows."""
    rng = np.random.default_rng(40 + s)
    A = rng.standard_normal((64, 40)) * (2.0 ** np.linspace(-540, 500, 64).round())[:, None]
    B = rng.standard_normal((40, 48)) * (2.0 ** np.linspace(-540, 500, 48).round())[None, :]
    A[5] = 0.0
    want = _want(A, B, "int8", s)
    assert np.any((want != 0) & (np.abs(want) < 2.0 ** -1022)) and np.any(np.abs(want) > 1e200)
    assert np.array_equal(_into(dmp, A, B, "int8", s, 0, 0), want)


def test_nan_rows_and_columns(dmp):
    rng = np.random.default_rng(50)
    A, B = rng.standard_normal((70, 50)), rng.standard_normal((50, 66))
    A[33, 7] = np.inf
    B[4, 65] = np.nan
    got = _into(dmp, A, B, "int8", 6, 0, 0)
    bad = np.zeros((70, 66), dtype=bool)
    bad[33, :] = bad[:, 65] = True
    assert np.all(np.isnan(got[bad]))
    A[33, 7], B[4, 65] = 0.0, 0.0
    ok = ~bad
    assert np.array_equal(got[ok], _want(A, B, "int8", 6)[ok])


@pytest.mark.parametrize("n", [160, 500, 1000, 1300, 2600])
def test_products_do_not_depend_on_how_tiles_are_shared(dmp, n):
    """Few tiles (parts of one tile on many CTAs), one partial wave whose planes
    stay in L2 and one whose planes do not: the bits of whole tiles."""
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    A = torch.randn((n, n), generator=g, device="cuda", dtype=torch.float64)
    prev = dmp.set_tc_split_tiles(True)
    try:
        a = dmp.ozaki_gemm(A, A, "int8", 6)
        dmp.set_tc_split_tiles(False)
        b = dmp.ozaki_gemm(A, A, "int8", 6)
    finally:
        dmp.set_tc_split_tiles(prev)
    assert torch.equal(a, b)
