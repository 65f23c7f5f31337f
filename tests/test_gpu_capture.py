"""The building blocks captured in a CUDA graph: launches that overlap the kernel before them
and clusters replay as they run directly, bit for bit, on new inputs too."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2602_03438_gb300 as P
    P.negf.load_library()
    return P


@pytest.mark.parametrize("prec,n,units", [("MIXED", 96, 3), ("MIXED", 128, 200), ("MIXED", 200, 2), ("MIXED", 300, 2),
                                          ("FP64", 40, 3), ("FP64", 64, 2), ("FP64", 128, 9)])
def test_products_and_inverses_replay(P, prec, n, units):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n + units)
    new = lambda: (torch.randn(units, n, n, dtype=torch.complex128, device="cuda", generator=gen) / n ** 0.5
                   + 2.0 * torch.eye(n, dtype=torch.complex128, device="cuda"))
    A, B = new(), new()
    X, D = torch.empty_like(A), torch.empty_like(A)
    ctx = P.Context(0, 1 << 30)
    p = getattr(P, prec)

    def chain():
        P.negf.negf_block_inverse(ctx, p, A, X)
        P.negf.negf_block_gemm(ctx, p, X, B, D, 0, 2, -1.0, 1.0, A)
        P.negf.negf_block_inverse(ctx, p, D, X)
    try:
        chain()
        assert ctx.sync() == 0
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            chain()
        for _ in range(2):
            A.copy_(new())
            B.copy_(new())
            chain()
            assert ctx.sync() == 0
            want = X.clone(), D.clone()
            X.zero_()
            D.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(X, want[0]) and torch.equal(D, want[1])
    finally:
        ctx.close()
