"""Hamiltonians that the set-up of a purification rejects, in the methods whose
steps are enqueued before the host has read the state."""

import pytest
import torch

from synth import make_hamiltonian

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,executor", [("fp64", "auto"), ("int8", "tc"), ("int8", "imma"), ("e4m3", "tc")])
@pytest.mark.parametrize("h", ["nan", "identity"])
def test_rejected_hamiltonian_runs_no_step(dmp, mode, executor, h):
    """A rejected H (NaN, or a multiple of the identity) stops the call before
    the first measure: no step may follow, and P holds the initial guess, which
    TRS4 and SP2 share, whatever the workspace held before."""
    n, n_occ = 200, 50
    if h == "nan":
        H = torch.from_numpy(make_hamiltonian(n, n_occ, seed=3).H).cuda()
        H[7, 100] = float("nan")
    else:
        H = 1.5 * torch.eye(n, dtype=torch.float64, device="cuda")
    code = dmp.ERR_NONFINITE if h == "nan" else dmp.ERR_INVALID_ARG
    opts = dmp.make_opts(mode, 7, executor)
    got = []
    for method, fill in (("sp2", 0), ("trs4", 0x3F), ("trs4", 0xBF)):
        ws = dmp.workspace(dmp.purify_workspace_bytes(n, opts)).fill_(fill)
        P = torch.full((n, n), 4.25, dtype=torch.float64, device="cuda")
        with pytest.raises(dmp.DmpError) as e:
            dmp.purify(H, n_occ, mode=mode, slices=7, executor=executor, method=method, P=P, ws=ws)
        assert e.value.code == code
        got.append(P.view(torch.int64))
    assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])
