"""Products with three group sums per element over several launches, in the area
that holds a whole wave of tiles and in the least one (other rounds of tiles).
The group sums are integers, so the results are the same bits, those of the int8
executor, and the oracle's."""

import numpy as np
import pytest
import torch

from oracle import ozaki as oz
from synth import make_hamiltonian

pytestmark = pytest.mark.gpu

RULE = {"int8": (7, "trunc"), "bf16": (8, "nearest"), "e4m3": (5, "nearest")}


# 152 and 240 tiles of 256 x 256, 130 in the least area only
@pytest.mark.parametrize("mode,s", [("int8", 9), ("int8", 10), ("bf16", 7), ("e4m3", 9)])
@pytest.mark.parametrize("m,n,k,wave", [(4700, 2000, 4100, True), (3840, 4096, 2048, True), (3300, 2500, 200, False)])
def test_products_in_either_area(dmp, mode, s, m, n, k, wave):
    g = torch.Generator(device="cuda")
    g.manual_seed(m + s)
    A = torch.randn((m, k), generator=g, device="cuda", dtype=torch.float64)
    B = torch.randn((k, n), generator=g, device="cuda", dtype=torch.float64)
    A *= 2.0 ** torch.randint(-20, 20, (m, 1), generator=g, device="cuda").double()
    most = dmp.gemm_workspace_bytes(m, n, k, mode, s)
    least = dmp.gemm_workspace_bytes(m, n, k, mode, s, least=True)
    assert most - least == (40 << 20 if wave and (mode != "e4m3" or k >= 4096) else 0)
    want = dmp.ozaki_gemm(A, B, mode, s, "tc", ws=dmp.workspace(least))
    assert torch.equal(dmp.ozaki_gemm(A, B, mode, s, "tc"), want)
    if mode == "int8":
        assert torch.equal(dmp.ozaki_gemm(A, B, mode, s, "imma"), want)
    rows, cols = [0, 255, 256, m // 2, m - 1], [0, 255, 511, n // 2 + 1, n - 1]
    beta, rounding = RULE[mode]
    ref = oz.ozaki_gemm(A.cpu().numpy()[rows], B.cpu().numpy()[:, cols], s, beta, rounding=rounding)
    assert np.array_equal(want.cpu().numpy()[np.ix_(rows, cols)], ref)


@pytest.mark.parametrize("mode,s", [("int8", 9), ("bf16", 7), ("e4m3", 9)])
@pytest.mark.parametrize("tile", [0, 256, 512])
def test_batches_in_either_area(dmp, mode, s, tile):
    ns = [2300, 900, 129, 1400]  # 45, 10, 1 and 21 tiles
    Hs = [torch.from_numpy(make_hamiltonian(n, n // 4, seed=n).H).cuda() for n in ns]
    o = dmp.make_opts(mode, s, "tc")
    most, least = dmp.batched_workspace_bytes(ns, o), dmp.batched_workspace_bytes(ns, o, least=True)
    assert most - least == 40 << 20
    prev = dmp.set_batched_tile(tile)
    try:
        ws = dmp.workspace(most)
        # one buffer of both lengths: a graph made for one is not taken for the other
        got = [dmp.purify_batched(Hs, [n // 4 for n in ns], mode=mode, slices=s, max_iter=6, ws=w,
                                  raise_on_error=False) for w in (ws, ws[:least], ws)]
    finally:
        dmp.set_batched_tile(prev)
    for Ps, infos, code in got[1:]:
        assert code == got[0][2] and infos == got[0][1]
        assert all(torch.equal(a, b) for a, b in zip(Ps, got[0][0]))
    with pytest.raises(dmp.DmpError) as e:
        dmp.purify_batched(Hs, [n // 4 for n in ns], mode=mode, slices=s, ws=ws[:least - 1])
    assert e.value.code == dmp.ERR_WORKSPACE
