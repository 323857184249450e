"""Calls whose memory does not hold the difference planes: the binding falls
back to the least workspace, and every result is the same, bit for bit."""

import pytest
import torch

from synth import make_hamiltonian

pytestmark = pytest.mark.gpu


@pytest.fixture
def no_room(dmp, monkeypatch):
    """Makes an allocation of more than `limit` bytes fail as a full GPU does."""
    real = dmp.workspace

    def limit(nbytes):
        def small(n, device=None):
            if n > nbytes:
                raise torch.cuda.OutOfMemoryError("no room")
            return real(n, device)

        monkeypatch.setattr(dmp, "workspace", small)

    return limit


N = 2000


@pytest.fixture(scope="module")
def H():
    return torch.from_numpy(make_hamiltonian(N, N // 4, seed=5).H).cuda()


def _same(fn, size, no_room):
    want = fn()
    no_room(size(least=True))
    got = fn()
    for a, b in zip(want, got):
        assert torch.equal(a, b) if isinstance(a, torch.Tensor) else a == b
    # and what does not fit either still fails
    no_room(size(least=True) - 1)
    with pytest.raises(torch.cuda.OutOfMemoryError):
        fn()


def test_purify(dmp, H, no_room):
    o = dmp.make_opts("int8", 5, refine=6)
    _same(lambda: dmp.purify(H, N // 4, slices=5, refine=6, max_iter=12),
          lambda least: dmp.purify_workspace_bytes(N, o, least=least), no_room)


def test_purify_host(dmp, H, no_room):
    o = dmp.make_opts("int8", 5)
    Hh = H.cpu()
    _same(lambda: dmp.purify_host(Hh, N // 4, slices=5, max_iter=12),
          lambda least: dmp.host_workspace_bytes(N, o, least=least), no_room)


def test_product(dmp, H, no_room):
    _same(lambda: (dmp.ozaki_gemm(H, H, "int8", 5),),
          lambda least: dmp.gemm_workspace_bytes(N, N, N, "int8", 5, least=least), no_room)


def test_expansion(dmp, H, no_room):
    o, p = dmp.make_opts("int8", 5), dmp.foe_params(0.2, 20, mu=0.0)
    _same(lambda: dmp.foe(H, 0.2, 20, mu=0.0, slices=5),
          lambda least: dmp.foe_workspace_bytes(N, p, o, least=least), no_room)


def test_backward(dmp, H, no_room):
    o = dmp.make_opts("int8", 6, max_iter=12)
    tape = torch.empty(dmp.tape_bytes(N, o), dtype=torch.uint8, device="cuda")
    P, _ = dmp.purify(H, N // 4, slices=6, max_iter=12, tape=tape)
    _same(lambda: (dmp.purify_backward(H, N // 4, tape, P, slices=6, max_iter=12),),
          lambda least: dmp.backward_workspace_bytes(N, o, least=least), no_room)
