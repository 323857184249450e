"""Purification steps that are enqueued before the host has read the state they
depend on: the elementwise SP2 / TRS4 step writes over its iterate, and every
step enqueued past the last one does nothing. The iterate P may have rows of any
length (nothing past column n is written) and any number of steps, and the result
does not depend on it, bit for bit. Sizes on both sides of the 1024 columns that
a block of the elementwise kernels takes."""

import pytest
import torch

from synth import make_hamiltonian

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["pm", "sp2", "trs4"])
@pytest.mark.parametrize("n,pad", [(33, 2), (130, 3), (1023, 1), (1026, 5)])
def test_padded_rows_give_the_same_bits(dmp, method, n, pad):
    H = torch.from_numpy(make_hamiltonian(n, n // 4, occ=(-2.0, -0.5), virt=(0.5, 2.0), seed=n).H).cuda()
    ref, info = dmp.purify(H, n // 4, mode="int8", slices=6, method=method)
    store = torch.full((n, n + pad), 7.0, dtype=torch.float64, device="cuda")
    _, info2 = dmp.purify(H, n // 4, mode="int8", slices=6, method=method, P=store[:, :n])
    assert info["status"] >= 0 and info["iters"] == info2["iters"] and info["energy"] == info2["energy"]
    assert torch.equal(store[:, :n], ref)
    assert (store[:, n:] == 7.0).all()


@pytest.mark.parametrize("method", ["pm", "sp2", "trs4"])
@pytest.mark.parametrize("max_iter", [1, 2, 3])
def test_a_run_cut_short_is_the_start_of_a_longer_one(dmp, method, max_iter):
    """The idempotency error of the last iterate, from P itself: no step past max_iter has touched it."""
    n = 130
    H = torch.from_numpy(make_hamiltonian(n, 30, occ=(-2.0, -0.5), virt=(0.5, 2.0), seed=7).H).cuda()
    P, info = dmp.purify(H, 30, mode="fp64", method=method, max_iter=max_iter)
    assert info["status"] == dmp.NOT_CONVERGED and info["iters"] == max_iter
    assert abs(torch.linalg.norm(P @ P - P).item() - info["idem"]) <= 1e-10
    assert abs(torch.trace(P).item() - info["trace"]) <= 1e-10
