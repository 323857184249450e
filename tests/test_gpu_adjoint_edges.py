"""The gradient at the edges of its kernels' 32 x 32 blocks and on both sides of
the rule that takes G P^2 and P G P as one product (digits of 42 bits and more)
or as two. Against the closed-form derivative of the spectral projector, with
the bound the ordinary sizes have (1e-6 of the largest entry)."""

import numpy as np
import pytest
import torch

from synth import make_hamiltonian, symmetric_gaussian
from test_gpu_adjoint import _dk, _gpu_grad

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,s", [("fp64", 7), ("int8", 6), ("e4m3", 8), ("e4m3", 9), ("bf16", 7)])
@pytest.mark.parametrize("n", [8, 31, 33, 65, 130])
def test_gradient_is_exact_and_symmetric(dmp, mode, s, n):
    n_occ = max(1, n // 4)
    h = make_hamiltonian(n, n_occ, occ=(-2.0, -0.25), virt=(0.25, 2.0), seed=n)
    W = symmetric_gaussian(n, seed=n + 1)
    _, G = _gpu_grad(dmp, h.H, n_occ, W, mode=mode, slices=s, executor="tc", tol=1e-10, checkpoint_every=3)
    dk = _dk(h.Q, h.e, n_occ, W)
    assert np.max(np.abs(G - dk)) <= 1e-6 * np.max(np.abs(dk))
    assert np.array_equal(G, G.T)
