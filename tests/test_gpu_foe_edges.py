"""dm_foe at the edges of its kernels' blocks, against the oracle.

Sizes about the 32 x 32 blocks of the elementwise kernels (one block, a block
and a row, odd sizes) and term counts about the groups of seven Frobenius
products (q = ceil(sqrt(M)) = 2, 8, 9, 10, 15). Bounds as in the tests of the
same quantities at ordinary sizes: 1e-12 for P at a given mu (coefficients and
accumulation round differently), 1e-11 for P and 1e-9 for mu when mu is solved
for. The output step of the recurrence reads and writes the running sum in
vectors where its alignment allows and element by element elsewhere: the same
bits."""

import numpy as np
import pytest
import torch

from oracle import foe as fo
from synth import make_hamiltonian

pytestmark = pytest.mark.gpu

BOUNDS = (-2.0, 2.0)


def _system(n):
    return make_hamiltonian(n, max(1, n // 4), occ=(-2.0, -0.3), virt=(0.3, 2.0), seed=n)


@pytest.mark.parametrize("scheme", ["recurrence", "ps"])
@pytest.mark.parametrize("n,M", [(2, 2), (31, 64), (33, 65), (65, 3), (130, 82)])
def test_given_mu(dmp, scheme, n, M):
    h = _system(n)
    ref, _ = fo.foe(h.H, 0.1, M, mu=0.05, bounds=BOUNDS, scheme=scheme)
    P, info = dmp.foe(torch.from_numpy(h.H).cuda(), 0.1, M, mu=0.05, bounds=BOUNDS, mode="fp64", scheme=scheme)
    P = P.cpu().numpy()
    assert info["status"] == dmp.OK
    assert np.max(np.abs(P - ref)) <= 1e-12
    assert np.array_equal(P, P.T)


@pytest.mark.parametrize("scheme", ["recurrence", "ps"])
@pytest.mark.parametrize("n,M", [(31, 64), (33, 65), (130, 82), (97, 200)])
def test_solved_mu(dmp, scheme, n, M):
    h = _system(n)
    n_occ = max(1, n // 4)
    ref, rinfo = fo.foe(h.H, 0.05, M, n_occ=n_occ, bounds=BOUNDS, scheme=scheme)
    P, info = dmp.foe(torch.from_numpy(h.H).cuda(), 0.05, M, n_occ=n_occ, bounds=BOUNDS, mode="fp64", scheme=scheme)
    assert info["status"] == dmp.OK
    assert abs(info["mu"] - rinfo["mu"]) <= 1e-9
    assert np.max(np.abs(P.cpu().numpy() - ref)) <= 1e-11


@pytest.mark.parametrize("mode,s", [("fp64", 1), ("int8", 7), ("e4m3", 8)])
@pytest.mark.parametrize("n,ldp,offset", [(130, 131, 0), (130, 132, 1), (257, 257, 1), (300, 300, 0)])
def test_running_sum_of_any_alignment(dmp, mode, s, n, ldp, offset):
    H = torch.from_numpy(_system(n).H).cuda()
    ref, _ = dmp.foe(H, 0.1, 20, mu=0.05, bounds=BOUNDS, mode=mode, slices=s)
    store = torch.full((offset + n * ldp,), 7.0, dtype=torch.float64, device="cuda")
    P = store[offset:].view(n, ldp)[:, :n]
    dmp.foe(H, 0.1, 20, mu=0.05, bounds=BOUNDS, mode=mode, slices=s, P=P)
    assert torch.equal(P, ref)
    assert (store[offset:].view(n, ldp)[:, n:] == 7.0).all() and (store[:offset] == 7.0).all()
