"""ozaki_gemm captured into a CUDA graph (its launches carry the programmatic
serialisation attribute, its area of group sums is cleared by a memset node and
handed from one replay to the next): replays on new inputs give the bits of the
direct call. Shared tiles of one launch, several rounds with digit differences,
three group sums per element over several rounds, and single-CTA tiles."""

import pytest
import torch

pytestmark = pytest.mark.gpu


def _fill(A, B, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    A.copy_(torch.randn(A.shape, generator=g, device="cuda", dtype=torch.float64))
    B.copy_(torch.randn(B.shape, generator=g, device="cuda", dtype=torch.float64))
    A[A.shape[0] // 2] *= 2.0 ** (seed % 40)


@pytest.mark.parametrize("m,n,k,mode,s", [(200, 130, 300, "int8", 5), (1000, 333, 257, "bf16", 6),
                                          (3900, 3800, 2600, "int8", 8), (2600, 2817, 2561, "int8", 5),
                                          (2700, 2600, 500, "e4m3", 9), (1500, 1500, 700, "fp64", 0)])
def test_replays_equal_the_direct_call(dmp, m, n, k, mode, s):
    A = torch.empty((m, k), dtype=torch.float64, device="cuda")
    B = torch.empty((k, n), dtype=torch.float64, device="cuda")
    C = torch.empty((m, n), dtype=torch.float64, device="cuda")
    ws = dmp.workspace(dmp.gemm_workspace_bytes(m, n, k, mode, s))
    _fill(A, B, 1)
    dmp.ozaki_gemm(A, B, mode, s, C=C, ws=ws)  # loads the device code
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        dmp.ozaki_gemm(A, B, mode, s, C=C, ws=ws)
    for seed in (2, 3, 3):
        _fill(A, B, seed)
        ws.fill_(0x5A)  # nothing may be taken over from an earlier call
        C.fill_(float("nan"))
        graph.replay()
        got = C.clone()
        assert torch.equal(got, dmp.ozaki_gemm(A, B, mode, s))
    # replays one after the other, without a wait between them
    _fill(A, B, 4)
    for _ in range(5):
        graph.replay()
    assert torch.equal(C, dmp.ozaki_gemm(A, B, mode, s))


def test_a_chain_of_captured_products(dmp):
    """Products that feed one another in one capture, on one workspace."""
    n = 600
    A = torch.empty((n, n), dtype=torch.float64, device="cuda")
    B = torch.empty_like(A)
    X, Y = torch.empty_like(A), torch.empty_like(A)
    ws = dmp.workspace(dmp.gemm_workspace_bytes(n, n, n, "int8", 6))
    _fill(A, B, 5)

    def chain():
        dmp.ozaki_gemm(A, B, "int8", 6, C=X, ws=ws)
        dmp.ozaki_gemm(X, A, "int8", 6, C=Y, ws=ws)
        dmp.ozaki_gemm(Y, B, "int8", 6, C=X, ws=ws)

    chain()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain()
    _fill(A, B, 6)
    graph.replay()
    got = X.clone(), Y.clone()
    chain()
    assert torch.equal(got[0], X) and torch.equal(got[1], Y)
