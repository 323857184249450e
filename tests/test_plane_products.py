"""The benchmark counts the plane products that the tensor cores form by the
library's rule for difference products. The rule shows in the workspaces: the
difference planes are what the least one leaves out."""

import pytest

import bench
from paper_2407_13299_gb300 import build


@pytest.mark.parametrize("mode,executor", [("int8", "tc"), ("int8", "imma"), ("bf16", "tc"), ("e4m3", "tc")])
def test_the_rate_counts_by_the_library_s_rule(mode, executor):
    build.build()
    from paper_2407_13299_gb300 import dmp

    up = lambda x, q: (x + q - 1) // q * q
    for n in (256, 1919, 1920, 2559, 2560, 8192):
        for k in range(1, 13 if mode == "e4m3" else 10):
            extra = (dmp.gemm_workspace_bytes(n, n, n, mode, k, executor) -
                     dmp.gemm_workspace_bytes(n, n, n, mode, k, executor, least=True))
            planes = extra // (2 * 2 * up(n, 256) * up(n, 128))  # bf16, both operands; 40 MiB may go with them
            saved = bench.pairs(k) - bench.plane_products_of(k, mode, executor, n)
            if mode == "int8" and executor == "tc":
                # a difference plane takes the place of two products; the squares of the digits below s come on top
                differences = sum(1 for i in range(1, k) for j in range(i + 1, k) if i + j <= k + 1)
                assert (saved > 0) == (planes >= 1)
                if saved > 0:
                    assert planes == differences
                    assert bench.plane_products_of(k, mode, executor, n) == k + 1 + differences
            else:
                assert saved == 0
