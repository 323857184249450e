"""The reverse step with one product V = (Y + Y^T / 2) P, Y = G P, in the place of
G P^2 and P G P (V + V^T = G P^2 + P G P + P^2 G): the same gradient exactly, and
to 1e-9 of it with digits of 42 bits and more, from which on dm_purify_backward
takes it (csrc/adjoint.cu). CPU, the oracle's products, one forward for both."""

from functools import partial

import numpy as np
import pytest

from oracle import adjoint as ad
from oracle import foe as fo
from oracle import ozaki as oz
from oracle import purify as pu
from synth import make_hamiltonian, symmetric_gaussian


def _sweep(h, fwd, W, product, merged):
    sym = fo.symmetric_output(product)
    G = 0.5 * (W + W.T)
    for k in range(fwd["iters"] - 1, -1, -1):
        P, c = fwd["iterates"][k], fwd["c_history"][k]
        X2 = sym(P, P)
        alpha, b2, b3, _ = pu.pm_weights(c)
        da, db2, db3 = ad.pm_weight_derivatives(c)
        Y = product(G, P)
        if merged:
            V = product(Y + 0.5 * Y.T, P)
            third = V + V.T
        else:
            YP, ZP = product(Y, P), product(Y.T, P)
            third = YP + YP.T + 0.5 * (ZP + ZP.T)
        td = np.trace(P) - np.trace(X2)
        tn = c * td
        dc = ((2.0 * P - 3.0 * X2) * td - tn * (np.eye(len(P)) - 2.0 * P)) / td**2
        dL_dc = np.sum(G * (da * P + db2 * X2)) + db3 * np.sum(Y * X2)
        G = alpha * G + b2 * (Y + Y.T) + b3 * third + dL_dc * dc
    return ad.initial_guess_adjoint(h.H, h.n_occ, fwd["init"], G, bounds_grad=False)


@pytest.mark.parametrize("s,beta,rounding,bound", [(None, None, None, 1e-12), (6, 7, "trunc", 1e-9),
                                                   (6, 8, "nearest", 1e-9), (9, 5, "nearest", 1e-9)])
def test_one_product_for_two(s, beta, rounding, bound):
    n = 150
    h = make_hamiltonian(n, n // 4, occ=(-2.0, -0.25), virt=(0.25, 2.0), seed=17)
    W = symmetric_gaussian(n, seed=18)
    product = pu.fp64_product if s is None else partial(oz.ozaki_gemm, s=s, beta=beta, rounding=rounding)
    fwd = pu.purify(h.H, h.n_occ, tol=1e-10, product=product, record=True)
    apart = _sweep(h, fwd, W, product, merged=False)
    merged = _sweep(h, fwd, W, product, merged=True)
    assert np.max(np.abs(apart - merged)) <= bound * np.max(np.abs(apart))
