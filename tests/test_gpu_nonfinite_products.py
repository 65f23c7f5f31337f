"""The sliced block products (the byte digits, and the call without a workspace) on operands with
infinities and NaN and on results past the range of a double.

A NaN or an infinity reaches every result of its row (or column); the other results are what they
are without it, bit for bit.  Scaling the operands by powers of two scales every digit image's
exponent and nothing else, so that the results scale bit for bit too, to infinity where the scaled
value has no double.
"""
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


def _product(P, A, B, way, op=(0, 0)):
    D = torch.empty_like(A)
    if way == "noalloc":
        n, u = A.shape[-1], A.shape[0]
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        P.negf.negf_block_gemm_noalloc(A, B, D, op[0], op[1], 1.0, 0.0, None, status=status)
        torch.cuda.synchronize()
        assert int(status) == 0
        return D
    ctx = P.Context(0, 1 << 28)
    try:
        P.negf.negf_block_gemm(ctx, P.MIXED, A, B, D, op[0], op[1], 1.0, 0.0, None)
        assert ctx.sync() == 0
    finally:
        ctx.close()
    return D


def _rand(n, units, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(units, n, n, dtype=torch.complex128, device="cuda", generator=g)


WAYS = [(16, "workspace"), (40, "workspace"), (128, "workspace"), (129, "workspace"), (300, "workspace"), (16, "noalloc"),
        (128, "noalloc"), (200, "noalloc")]


@pytest.mark.parametrize("n,way", WAYS)
@pytest.mark.parametrize("op", [(0, 0), (2, 2)])
def test_nonfinite_operands_reach_their_results(P, n, way, op):
    A, B = _rand(n, 4, n), _rand(n, 4, n + 1)
    clean = _product(P, A, B, way, op)
    i, j, k = n - 1, n // 2, n // 3
    nan, inf = complex(float("nan"), 0.0), complex(0.0, float("-inf"))

    def put(M, u, r, c, v, flip):
        M[u, c if flip else r, r if flip else c] = v

    put(A, 0, i, k, nan, op[0])       # unit 0: a NaN in row i of op(A)
    put(A, 1, i, k, inf, op[0])       # unit 1: an infinity there, and one in column j of op(B)
    put(B, 1, k, j, inf, op[1])
    put(B, 2, k, j, nan, op[1])       # unit 2: a NaN in column j of op(B); unit 3 stays
    D = _product(P, A, B, way, op)
    hit = torch.zeros(4, n, n, dtype=torch.bool, device="cuda")
    hit[0, i] = hit[1, i] = True
    hit[1, :, j] = hit[2, :, j] = True
    assert not bool(torch.isfinite(torch.view_as_real(D)).any(-1)[hit].any())
    assert torch.equal(D[~hit], clean[~hit])


@pytest.mark.parametrize("n,way", WAYS)
def test_results_past_the_range_become_infinite(P, n, way):
    A, B = _rand(n, 2, n), _rand(n, 2, n + 1)
    A[1, 0] = 0.0                     # zero results stay zero
    want = torch.view_as_real(_product(P, A, B, way))
    for ea, eb in ((500, 400), (512, 510), (900, 900), (900, -900), (-500, -400)):
        got = torch.view_as_real(_product(P, A * 2.0 ** ea, B * 2.0 ** eb, way))
        assert torch.equal(got, want * 2.0 ** (ea // 2 + eb // 2) * 2.0 ** (ea - ea // 2 + eb - eb // 2)), (ea, eb)
