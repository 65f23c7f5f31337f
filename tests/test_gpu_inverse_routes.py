"""Routes of the block inverses that the other tests' sizes do not take: the FP32 inverse in registers in
full rounds of 152 blocks, and zero columns in the FP64 inverse (one CTA per block, tiles launched
panel by panel, a cluster per block).

The tolerance is that of the other inverse tests, 8 n 2^-53 ||M||_F ||X||_F for I - M X.
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


def _invert(P, M, prec):
    units = M.shape[0]
    X = torch.empty_like(M)
    status = torch.zeros(units, dtype=torch.int32, device="cuda")
    ctx = P.Context(0, 1 << 30)
    try:
        P.negf.negf_block_inverse(ctx, prec, M, X, status)
        ctx.sync()
    finally:
        ctx.close()
    return X, status


def _matrix(n, units, seed):   # row interchanges in every panel
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    M = torch.randn(units, n, n, dtype=torch.complex128, device="cuda", generator=g) / n ** 0.5
    for u in range(units):
        M[u, torch.arange(n, device="cuda"), torch.randperm(n, device="cuda", generator=g)] += 2.0
    return M


def _check(M, X, skip=()):
    n = M.shape[-1]
    eye = torch.eye(n, dtype=M.dtype, device="cuda")
    for u in range(M.shape[0]):
        if u not in skip:
            bound = 8 * n * 2.0 ** -53 * float(M[u].norm()) * float(X[u].norm())
            assert float((eye - M[u] @ X[u]).norm()) <= bound, u


@pytest.mark.parametrize("n,units", [(97, 152), (100, 304), (128, 100), (128, 152), (128, 304)])
def test_registers_in_full_rounds(P, n, units):
    M = _matrix(n, units, n + units)
    X, status = _invert(P, M, P.MIXED)
    assert int(status.abs().sum()) == 0
    _check(M, X)


@pytest.mark.parametrize("n,units,col", [(30, 3, 29), (48, 120, 7), (40, 60, 39), (64, 3, 63), (64, 3, 0), (72, 9, 40),
                                         (100, 4, 98), (128, 3, 127), (128, 3, 64), (128, 20, 5), (200, 3, 199), (512, 2, 300)])
def test_zero_column_in_fp64(P, n, units, col):
    M = _matrix(n, units, n)
    M[1, :, col] = 0.0
    X, status = _invert(P, M, P.FP64)
    assert status.tolist() == [0, P.negf.NEGF_ERR_SINGULAR] + [0] * (units - 2)
    _check(M, X, skip=(1,))


@pytest.mark.parametrize("n,units", [(15, 160), (16, 152), (16, 153), (17, 200), (24, 153), (31, 160), (32, 96), (32, 97),
                                     (33, 3), (39, 96), (39, 153), (40, 130), (55, 120), (72, 100), (100, 160)])
def test_fp64_lines(P, n, units):
    M = _matrix(n, units, n + units)
    X, status = _invert(P, M, P.FP64)
    assert int(status.abs().sum()) == 0
    _check(M, X)


@pytest.mark.parametrize("n", [24, 40, 64, 100, 128])
def test_fp64_rounding(P, n):
    """No more rounding than a library inverse in the same precision: with one rounding of an entry's own
    size per step or per panel the mean residual of 20 blocks is that of torch.linalg.inv, up to a
    fifth for the order of operations (with two per step it is 1.2 to 1.9 times as large)."""
    M = _matrix(n, 20, 5 * n)
    X, _ = _invert(P, M, P.FP64)
    eye = torch.eye(n, dtype=M.dtype, device="cuda")
    mean = lambda Y: float((eye - M @ Y).flatten(1).norm(dim=1).mean())  # noqa: E731
    assert mean(X) <= 1.2 * mean(torch.linalg.inv(M))


@pytest.mark.parametrize("n,units,col", [(97, 152, 96), (128, 152, 127), (128, 152, 0), (128, 200, 64)])
def test_zero_column_in_registers_and_tiles(P, n, units, col):
    M = _matrix(n, units, n)
    M[1, :, col] = 0.0
    X, status = _invert(P, M, P.MIXED)
    assert status[1] == P.negf.NEGF_ERR_SINGULAR and int((status != 0).sum()) == 1
    _check(M, X, skip=(1,))
