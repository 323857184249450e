"""The two sizes of a workspace (host-side calls): the one a call runs fastest
in, which holds the planes of digit differences, and the least it needs."""

import pytest

from paper_2407_13299_gb300 import build


@pytest.fixture(scope="module")
def dmp():
    build.build()
    from paper_2407_13299_gb300 import dmp as binding

    return binding


def _up(x, q):
    return (x + q - 1) // q * q


def _sizes(dmp, entry, n, s, refine=0):
    o = dmp.make_opts("int8", s, "tc", refine=refine)
    if entry == "purify":
        f = lambda least: dmp.purify_workspace_bytes(n, o, least=least)
    elif entry == "host":
        f = lambda least: dmp.host_workspace_bytes(n, o, least=least)
    elif entry == "gemm":
        f = lambda least: dmp.gemm_workspace_bytes(n, n, n, "int8", s, "tc", least=least)
    elif entry == "backward":
        f = lambda least: dmp.backward_workspace_bytes(n, o, least=least)
    else:
        p = dmp.foe_params(0.1, 50, mu=0.0)
        f = lambda least: dmp.foe_workspace_bytes(n, p, o, least=least)
    return f(False), f(True)


# float64 matrices and operands' digit planes of each call beside 80 MiB of group sums
MATRICES = {"purify": 2, "host": 4, "gemm": 1, "backward": 6 + 2 * 8, "foe": 4}


@pytest.mark.parametrize("entry", sorted(MATRICES))
@pytest.mark.parametrize("n,s", [(1000, 7), (2000, 5), (3000, 8), (8192, 5), (20000, 9)])
def test_least_holds_the_digits_only(dmp, entry, n, s):
    most, least = _sizes(dmp, entry, n, s)
    digits = 2 * s * _up(n, 256) * _up(n, 128) * 2
    exact = MATRICES[entry] * 8 * n * n + digits + (80 << 20)
    # row sums (64 doubles a row), partial sums, exponents, coefficients of up to 16384 terms
    assert exact <= least <= exact + 64 * 8 * _up(n, 256) + (4 << 20)
    assert (most > least) == (n >= (1920 if s <= 6 else 2560))


@pytest.mark.parametrize("entry", sorted(MATRICES))
def test_no_workspace_grows_past_the_line(dmp, entry):
    line = 128 << 30
    for n in (25000, 40000, 50000, 66000):
        most, least = _sizes(dmp, entry, n, 5, refine=8 if entry in ("purify", "host") else 0)
        assert most <= max(least, line + (4 if entry == "host" else 0) * 4 * n * n)


def test_a_purification_that_fills_the_gpu_still_fits(dmp):
    """n = 65000, five slices refined with eight: H, P and the workspace take 64 n^2
    bytes (270 GB) without difference planes, 124 n^2 with them."""
    n = 65000
    most, least = _sizes(dmp, "purify", n, 5, refine=8)
    assert most == least and most + 2 * 8 * n * n < 284208 << 20


@pytest.mark.parametrize("mode,s,three", [("int8", 8, False), ("int8", 9, True), ("bf16", 6, False),
                                          ("bf16", 7, True), ("e4m3", 8, False), ("e4m3", 9, True)])
def test_three_group_sums_have_room_for_a_wave_of_tiles(dmp, mode, s, three):
    """Three sums per element of a 256 x 256 tile are 1.5 MiB, so 80 MiB hold the
    tiles of 53 of the GPU's 76 CTA pairs; 40 more hold a whole wave. A batch's
    tiles are walked whole, and it runs a quarter slower without."""
    wave = lambda size: size(False) - size(True)
    batch = lambda ns: wave(lambda least: dmp.batched_workspace_bytes(ns, dmp.make_opts(mode, s, "tc"), least))
    assert batch([4096, 4096]) == (three << 20) * 40
    assert batch([1024] * 5) == 0  # 50 tiles
    assert batch([1024] * 6) == (three << 20) * 40
    gemm = lambda m, n, k: wave(lambda least: dmp.gemm_workspace_bytes(m, n, k, mode, s, "tc", least))
    if mode == "int8":  # (beside the difference planes)
        return
    k = 4096 if mode == "e4m3" else 2048
    assert gemm(256 * 8, 256 * 19, k) == (three << 20) * 40
    assert gemm(256 * 8, 256 * 19, k - 1) == 0
    assert gemm(256 * 8, 256 * 18, k) == 0
