"""Difference products (diff_planes in csrc/dmp_internal.cuh): from a size on,
the INT8 mode multiplies (A_i - A_j)(B_i - B_j) instead of A_i B_j and A_j B_i.
The level sums are the same integers, so every result must be bit for bit that
of the pairs taken one by one -- which is what a call runs in a workspace that
has no room for the difference planes -- and of the int8 executor."""

import ctypes

import numpy as np
import pytest
import torch

from oracle import ozaki as oz

pytestmark = pytest.mark.gpu


def _plain_bytes(m, n, k, s):
    """ozaki_gemm's workspace without difference planes (256-byte pieces)."""
    up = lambda x, q: (x + q - 1) // q * q
    mp, np_, kp = up(m, 256), up(n, 256), up(k, 128)
    parts = [4 * mp, 4 * np_, 4, 2 * s * mp * kp, 2 * s * np_ * kp, 8 * n * k, 80 << 20]
    return sum(up(x, 256) for x in parts)


def _factors(m, n, k, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    A = torch.randn((m, k), generator=g, device="cuda", dtype=torch.float64)
    B = torch.randn((k, n), generator=g, device="cuda", dtype=torch.float64)
    # rows of very different sizes, zeros and entries of one sign
    A *= (2.0 ** torch.randint(-30, 30, (m, 1), generator=g, device="cuda").double())
    A[3], B[:, 5] = 0.0, 0.0
    A[7] = A[7].abs()
    return A, B


@pytest.mark.parametrize("s", [4, 5, 6, 7, 8, 9])
@pytest.mark.parametrize("m,n,k", [(2560, 2560, 2560), (2600, 2817, 2561)])
def test_equal_to_the_pairs_one_by_one(dmp, m, n, k, s):
    A, B = _factors(m, n, k, s)
    need, plain = dmp.gemm_workspace_bytes(m, n, k, "int8", s), _plain_bytes(m, n, k, s)
    assert plain < need
    got = dmp.ozaki_gemm(A, B, "int8", s)
    ws = dmp.workspace(plain)
    want = dmp.ozaki_gemm(A, B, "int8", s, ws=ws)
    assert torch.equal(got, want)
    # one byte less is refused, as before
    C = torch.empty_like(got)
    rc = dmp.lib().ozaki_gemm(m, n, k, A.data_ptr(), k, B.data_ptr(), n, C.data_ptr(), n, dmp.MODES["int8"], s,
                              dmp.EXECUTORS["tc"], ws.data_ptr(), plain - 1, ctypes.c_void_p(0))
    assert rc == dmp.ERR_WORKSPACE


@pytest.mark.parametrize("s,least", [(5, 1920), (8, 2560)])
def test_the_size_from_which_they_are_used(dmp, s, least):
    for n, used in ((least - 1, False), (least, True)):
        assert (dmp.gemm_workspace_bytes(n, n, n, "int8", s) > _plain_bytes(n, n, n, s)) == used
    # other digits, the int8 executor, and slice counts without a rule take none
    assert dmp.gemm_workspace_bytes(3000, 3000, 3000, "int8", 3) == _plain_bytes(3000, 3000, 3000, 3)
    assert dmp.gemm_workspace_bytes(3000, 3000, 3000, "bf16", 5) == _plain_bytes(3000, 3000, 3000, 5)


def test_against_the_int8_executor_and_the_oracle(dmp):
    n, s = 1920, 5
    A, B = _factors(n, n, n, 11)
    got = dmp.ozaki_gemm(A, B, "int8", s, "tc")
    assert torch.equal(got, dmp.ozaki_gemm(A, B, "int8", s, "imma"))
    rows, cols = [0, 3, 7, 1000, 1919], [0, 5, 640, 1918]
    a, b = A.cpu().numpy()[rows], B.cpu().numpy()[:, cols]
    assert np.array_equal(got.cpu().numpy()[np.ix_(rows, cols)], oz.ozaki_gemm(a, b, s, 7))
